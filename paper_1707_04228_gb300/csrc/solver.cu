// Solver context, setup, PCG driver and the C ABI (include/geneo_lam.h).
//
// Section 2.3: CG on P K u = P f (Eq. eq-pre) with P the two-level additive
// overlapping Schwarz preconditioner
//     P = Z K_0^{-1} Z^T + sum_j R_j^T A_j^{-1} R_j,
// A_j the Dirichlet matrices of the overlapping subdomains (direct solves),
// Z the GenEO coarse basis (Xi_j-weighted low-energy eigenvectors of the local
// Neumann matrices, Fig. eig), K_0 = Z^T K Z (dense Cholesky).
#include <algorithm>
#include <array>
#include <atomic>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <functional>
#include <initializer_list>
#include <mutex>
#include <thread>

#include "host_parallel.h"
#include "problem.h"
#include "slaves.h"

namespace gl {

void fail(int code, const std::string &msg) { throw Error{code, msg}; }

bool is_device_ptr(const void *p) {
    cudaPointerAttributes a{};
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

static thread_local std::string g_last_error;

// Inverse of a symmetric positive definite 6x6 matrix (Gauss-Jordan).
static void inv6(const double A[36], double X[36]) {
    double a[6][12];
    for (int i = 0; i < 6; ++i)
        for (int j = 0; j < 12; ++j) a[i][j] = j < 6 ? A[6 * i + j] : (j - 6 == i ? 1.0 : 0.0);
    for (int c = 0; c < 6; ++c) {
        int piv = c;
        for (int r = c + 1; r < 6; ++r)
            if (std::fabs(a[r][c]) > std::fabs(a[piv][c])) piv = r;
        if (std::fabs(a[piv][c]) < 1e-300) fail(GL_ERR_INVALID_ARG, "singular material compliance");
        if (piv != c)
            for (int j = 0; j < 12; ++j) std::swap(a[c][j], a[piv][j]);
        double d = a[c][c];
        for (int j = 0; j < 12; ++j) a[c][j] /= d;
        for (int r = 0; r < 6; ++r)
            if (r != c) {
                double f = a[r][c];
                for (int j = 0; j < 12; ++j) a[r][j] -= f * a[c][j];
            }
    }
    for (int i = 0; i < 6; ++i)
        for (int j = 0; j < 6; ++j) X[6 * i + j] = a[i][j + 6];
}

}  // namespace gl

using namespace gl;

namespace {
// Nested dissection stops at regions of at most this many nodes (fewer factor
// entries than larger leaves on the laminate subdomains: 66M against 83M per
// 6x9x92-element subdomain at 125).
constexpr int LEAF_NODES = 64;
std::atomic<long long> g_launches(0);   // kernels launched by gl_solve / gl_apply_* (hot path)
enum { PH_KU = 0, PH_LOCAL = 1, PH_COARSE = 2, PH_N = 3 };
struct Prof {
    bool on = false;
    bool levels = false;   // per-level sweep timing too (levels then run in sequence)
    cudaEvent_t ev[2 * PH_N] = {};
    double ms[PH_N] = {0, 0, 0};
    long long count[PH_N] = {0, 0, 0};
    int pending[PH_N] = {0, 0, 0};
};
}  // namespace

// A second stream on which the coarse correction of the preconditioner runs
// while the local sweeps run on the main one (both add into z atomically);
// fork/join events order it against the main stream (also inside a graph
// capture).  Created on first use with the owner's device current.
struct SideStream {
    cudaStream_t st = nullptr;
    cudaEvent_t fork = nullptr, join = nullptr;
    void ensure() {
        if (st) return;
        GL_CUDA(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking));
        GL_CUDA(cudaEventCreateWithFlags(&fork, cudaEventDisableTiming));
        GL_CUDA(cudaEventCreateWithFlags(&join, cudaEventDisableTiming));
    }
    ~SideStream() {
        if (fork) cudaEventDestroy(fork);
        if (join) cudaEventDestroy(join);
        if (st) cudaStreamDestroy(st);
    }
};

struct gl_ctx {
    Prof prof;
    int device = 0;
    cudaStream_t stream = 0;
    // materials (host, 36 per entry) and kind
    std::vector<double> matC;
    std::vector<uint8_t> mat_iso;
    bool have_mat = false, have_mesh = false, ready = false;
    MeshHost m;
    std::vector<double> psi_x;
    // device mesh data
    DBuf<double> d_tn, d_ln, d_rn, d_dr, d_X, d_C, d_geo, d_psi, d_theta, d_layer_angle, d_matC;
    DBuf<int> d_layer_of_ez, d_layer_mat, d_elem_mat;
    DBuf<uint8_t> d_resin, d_mask;   // resin elements; eliminated DOFs
    // boundary data
    std::vector<int64_t> dir_dof;
    std::vector<double> dir_val;
    DBuf<int64_t> d_dir_dof;
    DBuf<double> d_dir_val;
    std::vector<std::pair<int, std::array<double, 3>>> tractions;
    DBuf<double> d_ftrac;
    // solver
    gl_opts opts{};
    Problem prob;        // this laminate as a one-part problem (subdomain boxes, numbering)
    FactorPlan PD;       // local Dirichlet factors (all subdomains)
    DBuf<double> LD64;
    DBuf<float> LD32;
    Coarse co;           // GenEO coarse space and K_0^{-1}
    DBuf<double> cvec2;
    // work
    DBuf<double> x, r, z, p, q, ud, fe, partials, cvec, xl64;
    DBuf<double> ks;     // serendipity: the filled copy of K u's input
    int64_t n_dir = 0;   // entries of d_dir_dof / d_dir_val: the prescribed DOFs (and the serendipity slaves)
    DBuf<float> xl32;
    DBuf<CGScalars> S;
    DBuf<int> err;
    double *h_pin = nullptr;
    cudaEvent_t ev_scalar = nullptr;
    double ms_setup = 0;
    int64_t n_free = 0;
    SideStream side;

    ~gl_ctx() {
        if (h_pin) cudaFreeHost(h_pin);
        if (ev_scalar) cudaEventDestroy(ev_scalar);
    }
};

namespace {

int guard(const std::function<void()> &fn) {
    try {
        fn();
        return GL_OK;
    } catch (const Error &e) {
        g_last_error = e.msg;
        return e.code;
    } catch (const std::bad_alloc &) {
        g_last_error = "host out of memory";
        return GL_ERR_OOM;
    } catch (const std::exception &e) {
        g_last_error = e.what();
        return GL_ERR_CUDA;
    }
}

void require_ctx(gl_ctx *c) {
    if (!c) fail(GL_ERR_INVALID_ARG, "null context");
    GL_CUDA(cudaSetDevice(c->device));
}

// Copy n doubles between a caller's array (host or device) and device memory.
void to_device(double *dst, const double *src, int64_t n, cudaStream_t s) {
    if (n) GL_CUDA(cudaMemcpyAsync(dst, src, n * sizeof(double), cudaMemcpyDefault, s));
}
void from_device(double *dst, const double *src, int64_t n, cudaStream_t s) {
    if (n) GL_CUDA(cudaMemcpyAsync(dst, src, n * sizeof(double), cudaMemcpyDefault, s));
    GL_CUDA(cudaStreamSynchronize(s));
}

void check_err(gl_ctx *c, const char *what) {
    int h = 0;
    GL_CUDA(cudaMemcpyAsync(&h, c->err.p, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    GL_CUDA(cudaStreamSynchronize(c->stream));
    if (h) {
        c->err.zero(c->stream);
        if (h == 2) fail(GL_ERR_TIMEOUT, std::string(what) + ": a tensor-core wait gave up");
        fail(GL_ERR_NOT_SPD, std::string(what) + ": non-positive pivot");
    }
}

// *dst = *d (d in device memory), dst in host or device memory: what is enqueued
// so far is waited for, *pin is *d by then.
void finish_scalar(gl_ctx *c, double *dst, const double *d, const double *pin) {
    const bool on_device = dst && is_device_ptr(dst);
    if (on_device) to_device(dst, d, 1, c->stream);
    GL_CUDA(cudaStreamSynchronize(c->stream));
    if (dst && !on_device) *dst = *pin;
}

// An array of a caller: n doubles at p (p may be null).
struct Span {
    const double *p;
    int64_t n;
};

// Whether kernels of this context may use the caller's array in place: device
// memory of the context's device, aligned, all of it inside its allocation, and
// apart from the other arrays of the call (inputs that an in-place output must
// not overwrite early).  What may not goes through the work vectors by a copy,
// which refuses an array that is too short.
bool in_place(gl_ctx *c, Span a, std::initializer_list<Span> others = {}) {
    if (!a.p || (reinterpret_cast<uintptr_t>(a.p) & 7)) return false;
    for (const Span &o : others)
        if (o.p && a.p < o.p + o.n && o.p < a.p + a.n) return false;
    cudaPointerAttributes at{};
    if (cudaPointerGetAttributes(&at, a.p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice && at.device == c->device && in_device_span(a.p, a.n * sizeof(double));
}

// A displacement given by the caller as the stress kernels read it: in place,
// or through the work vector q (host memory, or constrained entries to fill).
const double *field_in(gl_ctx *c, const double *u) {
    const MeshHost &m = c->m;
    if (!has_slaves(m) && in_place(c, {u, m.n_dof})) return u;
    to_device(c->q.p, u, m.n_dof, c->stream);
    if (has_slaves(m)) slave_fill(m, c->q.p, c->stream);
    return c->q.p;
}

// Setup phase timing to stderr when GL_VERBOSE is set (syncs the stream).
void stamp(gl_ctx *c, const char *what) {
    static const bool on = std::getenv("GL_VERBOSE") != nullptr;
    static thread_local std::chrono::steady_clock::time_point last = std::chrono::steady_clock::now();
    if (!on) return;
    GL_CUDA(cudaStreamSynchronize(c->stream));
    auto now = std::chrono::steady_clock::now();
    size_t fr = 0, tot = 0;
    cudaMemGetInfo(&fr, &tot);
    std::fprintf(stderr, "[gl] %-34s %9.3f s   device used %.1f GB\n", what,
                 std::chrono::duration<double>(now - last).count(), (tot - fr) / 1e9);
    last = now;
}

// ---------------------------------------------------------------- geometry + material

void build_geometry(gl_ctx *c) {
    MeshHost &m = c->m;
    cudaStream_t s = c->stream;
    c->d_tn.upload(m.tn, s);
    c->d_ln.upload(m.ln, s);
    c->d_rn.upload(m.rn, s);
    c->d_X.alloc(3 * m.n_nodes);
    if (!m.node_dr.empty()) c->d_dr.upload(m.node_dr, s);
    else c->d_dr.release();
    launch_node_coords(m, c->d_tn.p, c->d_ln.p, c->d_rn.p, m.node_dr.empty() ? nullptr : c->d_dr.p, c->d_X.p, s);
    // serendipity: face and body centres at the serendipity interpolation of the element's nodes, so that
    // the Q2 geometry map of the element is its serendipity map
    if (m.element == 1) s20_fill(m, c->d_X.p, s);
    c->psi_x.assign(m.nx, 0.0);
    if (m.geometry == 1)
        for (int ex = 0; ex < m.nx; ++ex) {
            double tc = 0.5 * (m.sv[ex] + m.sv[ex + 1]);
            c->psi_x[ex] = std::min(std::max(tc, 0.0), 1.0) * m.arc_rad;
        }
    c->d_psi.upload(c->psi_x, s);
    c->d_layer_of_ez.upload(m.layer_of_ez, s);
    c->d_layer_mat.upload(m.layer_mat, s);
    c->d_layer_angle.upload(m.layer_angle, s);
    if (!m.theta.empty()) c->d_theta.upload(m.theta, s);
    else c->d_theta.release();
    if (!m.elem_mat.empty()) c->d_elem_mat.upload(m.elem_mat, s);
    else c->d_elem_mat.release();
    c->d_matC.upload(c->matC, s);
    c->d_C.alloc(36 * m.n_elem);
    launch_elem_material(m.n_elem, m.nx, m.ny, c->d_layer_of_ez.p, c->d_layer_mat.p, c->d_elem_mat.p,
                         c->d_layer_angle.p, c->d_theta.p, c->d_psi.p, c->d_matC.p, c->d_C.p, s);
    c->d_geo.alloc(270 * m.n_elem);
    launch_elem_geometry(m, c->d_X.p, c->d_geo.p, s);
    std::vector<uint8_t> resin(m.n_elem);
    for (int64_t e = 0; e < m.n_elem; ++e) {
        int ez = (int)(e / ((int64_t)m.nx * m.ny));
        resin[e] = c->mat_iso[m.elem_mat.empty() ? m.layer_mat[m.layer_of_ez[ez]] : m.elem_mat[e]];
    }
    c->d_resin.upload(resin, s);
    c->d_ftrac.alloc(m.n_dof);
    c->d_ftrac.zero(s);
    for (auto &t : c->tractions) launch_traction(m, c->d_X.p, t.first, t.second.data(), c->d_ftrac.p, s);
    if (has_slaves(m)) slave_fold(m, c->d_ftrac.p, s);            // f = P^T f_Q2
    GL_CUDA(cudaStreamSynchronize(s));
}

// ---------------------------------------------------------------- decomposition

// one start/stop pair; a pending pair is folded into the totals before reuse.
void prof_fold(gl_ctx *c, int ph) {
    Prof &P = c->prof;
    if (!P.pending[ph]) return;
    GL_CUDA(cudaEventSynchronize(P.ev[2 * ph + 1]));
    float ms = 0;
    GL_CUDA(cudaEventElapsedTime(&ms, P.ev[2 * ph], P.ev[2 * ph + 1]));
    P.ms[ph] += ms;
    P.count[ph] += 1;
    P.pending[ph] = 0;
}
void prof_begin(gl_ctx *c, int ph) {
    if (!c->prof.on) return;
    prof_fold(c, ph);
    GL_CUDA(cudaEventRecord(c->prof.ev[2 * ph], c->stream));
}
void prof_end(gl_ctx *c, int ph) {
    if (!c->prof.on) return;
    GL_CUDA(cudaEventRecord(c->prof.ev[2 * ph + 1], c->stream));
    c->prof.pending[ph] = 1;
}

int64_t factor_solve_launches(const FactorPlan &P) {
    int64_t n = 0;
    const bool halves = P.overlap_top > 0 && P.n_sub >= 2 && !P.clock.on;
    for (size_t d = 0; d < P.levels.size(); ++d) {
        const int64_t nf = (int64_t)P.levels[d].fronts.size(), na = P.half_fronts[d];
        if (halves) n += 2 * ((na > 0 ? 1 : 0) + (nf - na > 0 ? 1 : 0));
        else if (nf > 0) n += 2;
    }
    return n;
}

void apply_K(gl_ctx *c, const double *x, double *y, bool zeroed = false) {
    prof_begin(c, PH_KU);
    if (has_slaves(c->m)) {
        // constrained DOFs (serendipity, periodic width): y = P^T K_Q2 P x, the slave entries of x
        // filled in a copy and folded out of y
        GL_CUDA(cudaMemcpyAsync(c->ks.p, x, c->m.n_dof * sizeof(double), cudaMemcpyDeviceToDevice, c->stream));
        slave_fill(c->m, c->ks.p, c->stream);
        launch_ku(c->m, c->d_C.p, c->d_geo.p, c->ks.p, y, c->stream, zeroed);
        slave_fold(c->m, y, c->stream);
        g_launches += 2;
    } else {
        launch_ku(c->m, c->d_C.p, c->d_geo.p, x, y, c->stream, zeroed);
    }
    prof_end(c, PH_KU);
    g_launches += 1;
}

// z += sum_j R_j^T A_j^{-1} R_j r; xl holds three local vectors
template <class T>
void local_solve(const FactorPlan &P, const T *L, T *xl, const double *r, double *z, cudaStream_t s) {
    T *b = xl, *y = xl + P.n_local, *x = xl + 2 * P.n_local;
    gather_local<T>(P, r, b, y, x, s);
    factor_solve<T>(P, L, b, y, x, s);
    scatter_add_local<T>(P, x, z, s);
}

// z = M^{-1} r (r zero at Dirichlet DOFs; zeroed: z is zero already)
void apply_prec(gl_ctx *c, const double *r, double *z, bool zeroed = false) {
    cudaStream_t s = c->stream;
    if (!zeroed) GL_CUDA(cudaMemsetAsync(z, 0, c->m.n_dof * sizeof(double), s));
    // the coarse correction overlaps the local sweeps (whose upper dissection
    // levels leave SMs idle) unless the phases are being timed separately
    const bool side = c->co.n0 > 0 && !c->prof.on;
    if (side) {
        c->side.ensure();
        GL_CUDA(cudaEventRecord(c->side.fork, s));
        GL_CUDA(cudaStreamWaitEvent(c->side.st, c->side.fork, 0));
        coarse_apply(c->co, r, z, c->cvec.p, c->cvec2.p, c->side.st);
        GL_CUDA(cudaEventRecord(c->side.join, c->side.st));
        g_launches += 3;
    }
    prof_begin(c, PH_LOCAL);
    if (c->opts.precision == GL_PREC_MIXED) {
        local_solve<float>(c->PD, c->LD32.p, c->xl32.p, r, z, s);
    } else {
        local_solve<double>(c->PD, c->LD64.p, c->xl64.p, r, z, s);
    }
    prof_end(c, PH_LOCAL);
    g_launches += 2 + factor_solve_launches(c->PD);
    if (side) {
        GL_CUDA(cudaStreamWaitEvent(s, c->side.join, 0));
    } else if (c->co.n0 > 0) {
        prof_begin(c, PH_COARSE);
        coarse_apply(c->co, r, z, c->cvec.p, c->cvec2.p, s);
        prof_end(c, PH_COARSE);
        g_launches += 3;
    }
}

// Top levels of the overlapped two-half sweeps (0: sequential sweeps).  The
// default counts every level as top: the two halves sweep concurrently.
int sweep_overlap_top(const gl_opts &o) {
    if (o.sweep_overlap < 0) return 0;
    return o.sweep_overlap > 0 ? o.sweep_overlap : 1 << 20;
}

void setup(gl_ctx *c, const gl_opts &o) {
    auto t0 = std::chrono::steady_clock::now();
    if (!c->have_mat || !c->have_mesh) fail(GL_ERR_STATE, "gl_setup: materials and mesh must be set first");
    GL_REQUIRE(o.px >= 1 && o.py >= 1 && o.pz >= 1, "subdomain counts must be >= 1");
    GL_REQUIRE(o.overlap >= 1, "overlap must be >= 1");
    GL_REQUIRE(o.nev >= 0 && o.nev <= 28, "nev must be in [0, 28]");
    GL_REQUIRE(o.px <= c->m.nx && o.py <= c->m.ny && o.pz <= c->m.nz, "more subdomains than elements along an axis");
    GL_REQUIRE(!c->m.periodic || o.py == 1, "periodic width needs py = 1 (subdomains spanning the width)");
    GL_REQUIRE(o.precision == GL_PREC_FP64 || o.precision == GL_PREC_MIXED, "unknown precision mode");
    GL_REQUIRE(o.fp32_update == 0 || o.fp32_update == 1, "fp32_update must be 0 or 1");
    c->ready = false;
    c->opts = o;
    if (c->opts.max_iter <= 0) c->opts.max_iter = 2000;
    if (c->opts.tol <= 0) c->opts.tol = 1e-10;
    if (c->opts.resid_period <= 0) c->opts.resid_period = 50;
    cudaStream_t s = c->stream;
    const MeshHost &m = c->m;
    if (!c->err.p) {
        c->err.alloc(1);
        c->err.zero(s);
    }
    stamp(c, "start");
    build_geometry(c);
    stamp(c, "geometry, materials, loads");
    std::vector<uint8_t> is_dir(m.n_dof, 0);
    for (int64_t d : c->dir_dof) is_dir[d] = 1;
    {
        // the solver's eliminated DOFs: the prescribed ones with their values, and the slave
        // entries (serendipity centres, the periodic width plane) with 0 (a prescribed value
        // there is ignored: the constraint fixes it)
        std::vector<int64_t> dd(c->dir_dof);
        std::vector<double> dv(c->dir_val);
        if (has_slaves(m)) {
            std::vector<int64_t> sl = slave_dofs(m);
            std::vector<uint8_t> is_slave(m.n_dof, 0);
            for (int64_t d : sl) is_slave[d] = 1;
            dd.clear();
            dv.clear();
            size_t k = 0;
            for (int64_t d = 0; d < m.n_dof; ++d) {
                while (k < c->dir_dof.size() && c->dir_dof[k] < d) ++k;
                const bool pres = k < c->dir_dof.size() && c->dir_dof[k] == d;
                if (is_slave[d]) {
                    dd.push_back(d);
                    dv.push_back(0.0);
                    is_dir[d] = 1;
                } else if (pres) {
                    dd.push_back(d);
                    dv.push_back(c->dir_val[k]);
                }
            }
        }
        c->d_dir_dof.upload(dd, s);
        c->d_dir_val.upload(dv, s);
        c->n_dir = (int64_t)dd.size();
        c->d_mask.upload(is_dir, s);
        GL_CUDA(cudaStreamSynchronize(s));   // the lists are released at the end of this scope
    }
    c->n_free = m.n_dof - (int64_t)std::count(is_dir.begin(), is_dir.end(), (uint8_t)1);
    // the laminate as a one-part problem
    Problem &P = c->prob;
    P = Problem();
    P.stream = s;
    P.d_err = c->err.p;
    P.n_dof = m.n_dof;
    P.n_elem = m.n_elem;
    P.C = c->d_C.p;
    P.geo = c->d_geo.p;
    P.stamp = [c](const char *w) { stamp(c, w); };
    part_boxes(m, c->opts.px, c->opts.py, c->opts.pz, c->opts.overlap, P.boxes);
    {
        Part pt;
        pt.m = &c->m;
        pt.is_dir = is_dir;
        pt.sub0 = 0;
        pt.sub1 = (int)P.boxes.size();
        P.parts.push_back(std::move(pt));
    }
    P.sub_part.assign(P.boxes.size(), 0);
    {
        std::vector<SubSymbolic> syms;
        problem_symbolic(P, false, LEAF_NODES, syms);
        build_plan(syms, c->PD, s);
    }
    c->PD.ws_budget_bytes = c->opts.factor_ws_bytes > 0 ? c->opts.factor_ws_bytes : 6e9;
    c->PD.tc_update = c->opts.fp32_update == 0;
    c->PD.overlap_top = sweep_overlap_top(c->opts);
    c->PD.s20 = m.element == 1;
    stamp(c, "Dirichlet symbolic");
    if (std::getenv("GL_VERBOSE")) {
        // per dissection level: fronts, factor nonzeros the sweeps touch, the largest front
        for (size_t dpt = 0; dpt < c->PD.levels.size(); ++dpt) {
            const Level &Lv = c->PD.levels[dpt];
            double ent = 0, emax = 0;
            for (int g : Lv.fronts) {
                const FrontDesc &d = c->PD.fr[g];
                const double e = 0.5 * d.p * (d.p + 1.0) + (double)d.p * d.q;
                ent += e;
                emax = std::max(emax, e);
            }
            std::fprintf(stderr, "[gl]   level %2zu: %7zu fronts, %9.3e entries, largest %9.3e, max_f %d\n", dpt,
                         Lv.fronts.size(), ent, emax, Lv.max_f);
        }
    }
    // the Neumann matrices' symbolic phase runs on host threads while the device factors the Dirichlet ones
    std::future<std::vector<SubSymbolic>> neumann;
    if (c->opts.nev > 0) neumann = neumann_symbolic(P, LEAF_NODES);
    if (c->opts.precision == GL_PREC_MIXED) {
        c->LD64.release();
        c->LD32.alloc(c->PD.l_size);
        numeric_factor<float>(c->PD, c->d_C.p, c->d_geo.p, nullptr, 0.0, c->LD32.p, c->err.p, s);
    } else {
        c->LD32.release();
        c->LD64.alloc(c->PD.l_size);
        numeric_factor<double>(c->PD, c->d_C.p, c->d_geo.p, nullptr, 0.0, c->LD64.p, c->err.p, s);
    }
    check_err(c, "local Dirichlet factorisation");
    stamp(c, "Dirichlet factorisation");
    c->co = Coarse();
    if (c->opts.nev > 0) problem_coarse(P, c->opts, c->PD, neumann.get(), c->co);
    if (std::getenv("GL_VERBOSE"))
        std::fprintf(stderr, "[gl] GenEO block steps (max over groups): %d\n", c->co.eig_iters);
    stamp(c, "GenEO coarse space + K0");
    if (c->co.n_dropped && std::getenv("GL_VERBOSE"))
        std::fprintf(stderr, "[gl]   %d dependent coarse columns dropped\n", c->co.n_dropped);
    // work vectors
    const int64_t N = m.n_dof;
    if (has_slaves(m)) c->ks.alloc(N);
    else c->ks.release();
    for (DBuf<double> *b : {&c->x, &c->r, &c->z, &c->p, &c->q, &c->ud, &c->fe}) b->alloc(N);
    c->partials.alloc(RED_SCRATCH);
    c->partials.zero(s);
    c->cvec.alloc(std::max(1, c->co.n0));
    c->cvec2.alloc(std::max(1, c->co.n0));
    if (c->opts.precision == GL_PREC_MIXED) {
        c->xl32.alloc(3 * c->PD.n_local);
        c->xl64.release();
    } else {
        c->xl64.alloc(3 * c->PD.n_local);
        c->xl32.release();
    }
    c->S.alloc(1);
    if (!c->h_pin) GL_CUDA(cudaMallocHost(&c->h_pin, 8 * sizeof(double)));
    if (!c->ev_scalar) GL_CUDA(cudaEventCreateWithFlags(&c->ev_scalar, cudaEventDisableTiming));
    GL_CUDA(cudaStreamSynchronize(s));
    if (c->prof.levels) level_clock_enable(c->PD, true);
    c->ready = true;
    c->ms_setup = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
}

// The scalar's way to the host, and the host's wait for it; what is enqueued in
// between runs meanwhile.
void send_scalar(gl_ctx *c, const double *d) {
    GL_CUDA(cudaMemcpyAsync(c->h_pin, d, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    GL_CUDA(cudaEventRecord(c->ev_scalar, c->stream));
}
double await_scalar(gl_ctx *c) {
    GL_CUDA(cudaEventSynchronize(c->ev_scalar));
    return c->h_pin[0];
}

double read_scalar(gl_ctx *c, const double *d) {
    GL_CUDA(cudaMemcpyAsync(c->h_pin, d, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    GL_CUDA(cudaStreamSynchronize(c->stream));
    return c->h_pin[0];
}

// Effective right-hand side fe = f - K u_D on the free DOFs, 0 on Dirichlet DOFs.
void prepare_rhs(gl_ctx *c, const double *f, bool homogeneous) {
    cudaStream_t s = c->stream;
    const int64_t N = c->m.n_dof, nd = c->n_dir;
    if (f) to_device(c->fe.p, f, N, s);
    else GL_CUDA(cudaMemcpyAsync(c->fe.p, c->d_ftrac.p, N * sizeof(double), cudaMemcpyDeviceToDevice, s));
    c->ud.zero(s);
    if (!homogeneous) set_entries(c->ud.p, c->d_dir_dof.p, nd, c->d_dir_val.p, s);
    apply_K(c, c->ud.p, c->q.p);
    sub(c->fe.p, c->fe.p, c->q.p, N, s);
    set_entries(c->fe.p, c->d_dir_dof.p, nd, nullptr, s);
    g_launches += 1 + (nd ? 2 : 0);
}

// r = fe - K x on the free DOFs in FP64, r.r -> S->rr
void true_residual(gl_ctx *c, CGScalars *S) {
    apply_K(c, c->x.p, c->q.p);
    set_entries(c->q.p, c->d_dir_dof.p, c->n_dir, nullptr, c->stream);
    sub(c->r.p, c->fe.p, c->q.p, c->m.n_dof, c->stream);
    dot(c->r.p, c->r.p, c->m.n_dof, c->partials.p, &S->rr, c->stream);
    g_launches += (c->n_dir ? 1 : 0) + 2;
}

// PCG solve of K u = f into u (or left in c->x when u is that vector);
// homogeneous = zero Dirichlet values (adjoint solves).
void solve(gl_ctx *c, const double *f, double *u, gl_info *info, bool homogeneous = false) {
    if (!c->ready) fail(GL_ERR_STATE, "gl_solve before gl_setup");
    cudaStream_t s = c->stream;
    const int64_t N = c->m.n_dof, nd = c->n_dir;
    cudaEvent_t e0, e1;
    GL_CUDA(cudaEventCreate(&e0));
    GL_CUDA(cudaEventCreate(&e1));
    GL_CUDA(cudaEventRecord(e0, s));
    prepare_rhs(c, f, homogeneous);
    CGScalars *S = c->S.p;
    c->S.zero(s);
    dot(c->fe.p, c->fe.p, N, c->partials.p, &S->ff, s);
    const int nds = nd ? 1 : 0;   // set_entries launches a kernel only for a non-empty list
    g_launches += 1;
    const double ff = read_scalar(c, &S->ff);
    if (!std::isfinite(ff)) {
        GL_CUDA(cudaEventDestroy(e0));
        GL_CUDA(cudaEventDestroy(e1));
        fail(GL_ERR_NAN, "non-finite load vector");
    }
    const bool mixed = c->opts.precision == GL_PREC_MIXED;
    c->x.zero(s);
    GL_CUDA(cudaMemcpyAsync(c->r.p, c->fe.p, N * sizeof(double), cudaMemcpyDeviceToDevice, s));
    int iters = 0, status = GL_OK;
    double rel = 0.0;
    if (ff > 0.0) {
        apply_prec(c, c->r.p, c->z.p);
        dot(c->r.p, c->z.p, N, c->partials.p, &S->rho, s);
        g_launches += 1;
        GL_CUDA(cudaMemcpyAsync(c->p.p, c->z.p, N * sizeof(double), cudaMemcpyDeviceToDevice, s));
        rel = 1.0;
        // z = M r, beta and the next direction (q zeroed for the next K p)
        auto next_direction = [&]() {
            if (mixed) {
                dot(c->r.p, c->z.p, N, c->partials.p, &S->rz_old, s);   // flexible beta
                g_launches += 1;
            }
            apply_prec(c, c->r.p, c->z.p, !mixed);
            dot(c->r.p, c->z.p, N, c->partials.p, &S->rho_new, s);
            cg_update_p(c->p.p, c->z.p, c->q.p, N, S, c->partials.p, s);
            g_launches += 2;
        };
        for (int it = 1; it <= c->opts.max_iter; ++it) {
            apply_K(c, c->p.p, c->q.p, it > 1);
            dot(c->p.p, c->q.p, N, c->partials.p, &S->pq, s);   // p is zero at the eliminated DOFs
            cg_update_xr(c->x.p, c->r.p, c->p.p, c->q.p, c->d_mask.p, mixed ? nullptr : c->z.p, N, S, c->partials.p, s);
            g_launches += 2;
            // The host waits for ||r||; as long as the last one was far from the tolerance the next direction is
            // enqueued first and the device does not wait with it (if the iteration does end here after all, that
            // direction is not used).
            const bool special = mixed && it % c->opts.resid_period == 0;
            const bool ahead = rel > 100.0 * c->opts.tol && it < c->opts.max_iter && !special;
            send_scalar(c, &S->rr);
            if (ahead) next_direction();
            const double rr = await_scalar(c);
            iters = it;
            if (!std::isfinite(rr)) {
                status = GL_ERR_NAN;
                break;
            }
            rel = std::sqrt(rr / ff);
            // FP64: stop on the recurrence residual; the FP64 true residual is reported after the
            // loop (on these laminates its rounding floor lies near 1e-10 * ||K|| ||x|| / ||f||).
            // Mixed: the FP32 preconditioner lets the recurrence drift from the true residual, so
            // a passing recurrence is confirmed on r = fe - K x in FP64; if that misses tol, r
            // is replaced by it and the iteration goes on.
            bool replaced = false;
            if (rel <= c->opts.tol) {
                if (!mixed) break;
                true_residual(c, S);
                const double rt = read_scalar(c, &S->rr);
                if (!std::isfinite(rt)) {
                    status = GL_ERR_NAN;
                    break;
                }
                rel = std::sqrt(rt / ff);
                if (rel <= c->opts.tol) break;
                replaced = true;
            }
            if (it == c->opts.max_iter) {
                status = GL_ERR_NOT_CONVERGED;
                break;
            }
            if (special && !replaced) {
                // residual replacement: r = fe - K x in FP64
                apply_K(c, c->x.p, c->q.p);
                set_entries(c->q.p, c->d_dir_dof.p, nd, nullptr, s);
                sub(c->r.p, c->fe.p, c->q.p, N, s);
                g_launches += nds + 1;
            }
            if (replaced && ahead) {
                // a fall by more than 100 onto a residual that does not hold: z, p and rho are those of the
                // recurrence's next step, so the directions start anew from the true residual
                apply_prec(c, c->r.p, c->z.p);
                dot(c->r.p, c->z.p, N, c->partials.p, &S->rho, s);
                GL_CUDA(cudaMemcpyAsync(c->p.p, c->z.p, N * sizeof(double), cudaMemcpyDeviceToDevice, s));
                c->q.zero(s);
                g_launches += 1;
            } else if (!ahead) {
                next_direction();
            }
        }
    }
    // true residual and the full displacement
    true_residual(c, S);
    const double rt = read_scalar(c, &S->rr);
    axpy(c->x.p, 1.0, c->ud.p, N, s);
    g_launches += 1;
    if (has_slaves(c->m)) {
        slave_fill(c->m, c->x.p, s);   // the constrained entries carry the field's values
        g_launches += 1;
    }
    for (int ph = 0; ph < PH_N; ++ph) prof_fold(c, ph);
    GL_CUDA(cudaEventRecord(e1, s));
    if (u != c->x.p) to_device(u, c->x.p, N, s);
    GL_CUDA(cudaStreamSynchronize(s));
    float ms = 0;
    GL_CUDA(cudaEventElapsedTime(&ms, e0, e1));
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (info) {
        info->iters = iters;
        info->status = status;
        info->rel_resid = rel;
        info->rel_resid_true = ff > 0 ? std::sqrt(rt / ff) : 0.0;
        info->ms_setup = c->ms_setup;
        info->ms_solve = ms;
        info->n_free = c->n_free;
        info->n_coarse = c->co.n0;
        info->n_coarse_dropped = c->co.n_dropped;
        info->factor_nnz = c->PD.l_size;
    }
    if (status != GL_OK) {
        g_last_error = status == GL_ERR_NAN ? "NaN/Inf in the PCG iteration" : "PCG reached max_iter";
        throw Error{status, g_last_error};
    }
}

}  // namespace

// ====================================================================== many laminates at once

struct gl_batch {
    int device = 0;
    cudaStream_t stream = 0;
    bool own_stream = false, ready = false;
    std::vector<gl_ctx *> items;
    std::vector<cudaStream_t> item_streams;   // each laminate's own stream, given back on destruction
    gl_opts opts{};
    Problem prob;
    FactorPlan PD;
    DBuf<double> LD64;
    DBuf<float> LD32;
    Coarse co;
    std::vector<PartDesc> parts;
    DBuf<PartDesc> d_parts;
    std::vector<std::array<int, 2>> grid;     // (px, py) per laminate
    std::vector<int64_t> n_free;
    int64_t N = 0, E = 0, ndir = 0;
    DBuf<double> C, geo, f, x, r, z, p, q, ud, fe, c1, c2, xl64, partials, scal;
    DBuf<float> xl32;
    DBuf<int> ints;                           // active (n), iters (n), n_active (1)
    DBuf<int64_t> d_dir;
    DBuf<double> d_dirval;
    DBuf<int> err;
    int *h_active = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t gexec = nullptr;
    double ms_setup = 0;
    SideStream side;
    ~gl_batch() {
        if (gexec) cudaGraphExecDestroy(gexec);
        if (graph) cudaGraphDestroy(graph);
        if (h_active) cudaFreeHost(h_active);
        for (size_t i = 0; i < item_streams.size(); ++i) items[i]->stream = item_streams[i];
        if (own_stream) cudaStreamDestroy(stream);
    }
    SegScalars seg() {
        const int n = (int)items.size();
        return SegScalars{scal.p, scal.p + n, scal.p + 2 * n, scal.p + 3 * n, scal.p + 4 * n, scal.p + 5 * n,
                          ints.p, ints.p + n};
    }
};

namespace {

// Decomposition autotuner: candidates are in-plane grids (px, py, 1) with
// 8 <= px py <= 64 whose element boxes have an aspect ratio within [1/2, 2]
// (all of them if none qualifies).  For each, the symbolic factorisation of
// the central subdomain gives factor entries and factorisation flops, scaled
// by the subdomain count; the predicted time of one solve is
//   setup = (Dirichlet flops + 2x for the Neumann factor) / F
//         + 50 nev eigensolver solves x 4 flops x 1.6 nnz / F
//         + (2 n0)^3 / 3 / F                     (coarse inverse)
//   iteration = max(16 nnz / B, 4 nnz / F)       (FP64 sweeps; 8 nnz / B mixed)
//   total = setup + 40 iterations,
// with F = 0.8e12 flop/s (FP64) and B = 4.5e12 B/s (sustained HBM); the ratios
// Neumann/Dirichlet (1.6x entries, 2x flops) were measured on the corner laminate.
// The set-up terms are those of products on the FP64 pipe and of a subspace
// iteration.  The products run on the tensor cores now and the block Krylov
// method takes some 14 steps of eight solves, so set-up is priced too high and
// the choice leans to smaller factors than the fastest total would have.
std::vector<std::array<int, 2>> autotune_candidates(const MeshHost &m) {
    std::vector<std::array<int, 2>> cands, all;
    for (int px = 1; px <= std::min(64, m.nx); ++px)
        for (int py = 1; py <= std::min(64, m.ny); ++py) {
            const int ns = px * py;
            if (ns < 8 || ns > 64) continue;
            all.push_back({px, py});
            const double ax = (double)m.nx / px, ay = (double)m.ny / py;
            if (ax <= 2 * ay && ay <= 2 * ax) cands.push_back({px, py});
        }
    if (cands.empty()) cands = all;
    return cands;
}

double autotune_cost(const MeshHost &m, const std::vector<uint8_t> &is_dir, int overlap, int nev, bool mixed,
                     std::array<int, 2> cd) {
    const double F = 0.8e12, B = 4.5e12;
    const int px = cd[0], py = cd[1];
    std::vector<SubBox> boxes;
    part_boxes(m, px, py, 1, overlap, boxes);
    SubSymbolic S;
    build_symbolic(m, boxes[(py / 2) * px + px / 2], is_dir, false, LEAF_NODES, S);
    const int ns = px * py;
    double fl = 0.0;
    for (const Supernode &sn : S.sn) {
        const double f = sn.p + sn.q;
        for (int j = 0; j < sn.p; ++j) fl += (f - j) * (f - j);
    }
    const double nnz = (double)S.l_size * ns, flops = fl * ns, n0 = (double)ns * nev;
    const double setup = (mixed ? 0.1 : 1.0) * flops / F + 2.0 * flops / F + 25.0 * 2 * nev * 4.0 * 1.6 * nnz / F +
                         8.0 * n0 * n0 * n0 / 3.0 / F;
    const double iter = mixed ? 8.0 * nnz / B : std::max(16.0 * nnz / B, 4.0 * nnz / F);
    return setup + 40.0 * iter;
}

// The grid of every laminate: its candidates' costs on all host threads, the
// first of the cheapest taken.
void autotune_grids(const std::vector<gl_ctx *> &items, const std::vector<std::vector<uint8_t>> &is_dir, int overlap,
                    int nev, bool mixed, std::vector<std::array<int, 2>> &grid) {
    const int n = (int)items.size();
    std::vector<std::vector<std::array<int, 2>>> cands(n);
    std::vector<std::pair<int, int>> jobs;
    for (int i = 0; i < n; ++i) {
        cands[i] = autotune_candidates(items[i]->m);
        for (int k = 0; k < (int)cands[i].size(); ++k) jobs.push_back({i, k});
    }
    std::vector<double> cost(jobs.size());
    parallel_for((int)jobs.size(), [&](int q) {
        const int i = jobs[q].first;
        cost[q] = autotune_cost(items[i]->m, is_dir[i], overlap, nev, mixed, cands[i][jobs[q].second]);
    });
    std::vector<double> best(n, 1e300);
    for (int i = 0; i < n; ++i)
        grid[i] = cands[i].empty() ? std::array<int, 2>{std::min(items[i]->m.nx, 2), std::min(items[i]->m.ny, 2)}
                                   : cands[i][0];
    for (size_t q = 0; q < jobs.size(); ++q)
        if (cost[q] < best[jobs[q].first]) {
            best[jobs[q].first] = cost[q];
            grid[jobs[q].first] = cands[jobs[q].first][jobs[q].second];
        }
}

__global__ void k_seg_init(SegScalars S, int n) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    S.iters[i] = 0;
    S.active[i] = S.ff[i] > 0.0 ? 1 : 0;
    S.rz_old[i] = 0.0;
}

void batch_precond(gl_batch *b, const double *r, double *z) {
    cudaStream_t s = b->stream;
    GL_CUDA(cudaMemsetAsync(z, 0, b->N * sizeof(double), s));
    // coarse correction on the side stream, overlapping the local sweeps
    const bool side = b->co.n0 > 0;
    if (side) {
        b->side.ensure();
        GL_CUDA(cudaEventRecord(b->side.fork, s));
        GL_CUDA(cudaStreamWaitEvent(b->side.st, b->side.fork, 0));
        coarse_apply(b->co, r, z, b->c1.p, b->c2.p, b->side.st);
        GL_CUDA(cudaEventRecord(b->side.join, b->side.st));
        g_launches += 3;
    }
    if (b->opts.precision == GL_PREC_MIXED) {
        local_solve<float>(b->PD, b->LD32.p, b->xl32.p, r, z, s);
    } else {
        local_solve<double>(b->PD, b->LD64.p, b->xl64.p, r, z, s);
    }
    g_launches += 2 + factor_solve_launches(b->PD);
    if (side) GL_CUDA(cudaStreamWaitEvent(s, b->side.join, 0));
}

void batch_ku(gl_batch *b, const double *x, double *y) {
    launch_ku_batch(b->d_parts.p, (int)b->parts.size(), b->E, b->N, b->C.p, b->geo.p, x, y, b->stream);
    g_launches += 1;
}

void batch_setup(gl_batch *b, const gl_opts &o) {
    auto t0 = std::chrono::steady_clock::now();
    GL_REQUIRE(o.overlap >= 1, "overlap must be >= 1");
    GL_REQUIRE(o.nev >= 0 && o.nev <= 28, "nev must be in [0, 28]");
    GL_REQUIRE(o.precision == GL_PREC_FP64 || o.precision == GL_PREC_MIXED, "unknown precision mode");
    GL_REQUIRE(o.fp32_update == 0 || o.fp32_update == 1, "fp32_update must be 0 or 1");
    b->ready = false;
    b->opts = o;
    if (b->opts.max_iter <= 0) b->opts.max_iter = 2000;
    if (b->opts.tol <= 0) b->opts.tol = 1e-10;
    if (b->opts.resid_period <= 0) b->opts.resid_period = 50;
    cudaStream_t s = b->stream;
    const int n = (int)b->items.size();
    if (!b->err.p) {
        b->err.alloc(1);
        b->err.zero(s);
    }
    // geometry and loads of every laminate, on the batch stream
    b->parts.clear();
    b->N = b->E = 0;
    std::vector<std::vector<uint8_t>> is_dir(n);
    b->n_free.assign(n, 0);
    for (int i = 0; i < n; ++i) {
        gl_ctx *c = b->items[i];
        if (!c->have_mat || !c->have_mesh) fail(GL_ERR_STATE, "batch: every laminate needs materials and a mesh");
        c->stream = s;
        build_geometry(c);
        const MeshHost &m = c->m;
        PartDesc pd{};
        pd.elem_off = b->E;
        pd.dof_off = b->N;
        pd.n_dof = m.n_dof;
        pd.nx = m.nx;
        pd.ny = m.ny;
        pd.NX = m.NX;
        pd.NY = m.NY;
        b->parts.push_back(pd);
        b->N += m.n_dof;
        b->E += m.n_elem;
        is_dir[i].assign(m.n_dof, 0);
        for (int64_t d : c->dir_dof) is_dir[i][d] = 1;
        b->n_free[i] = m.n_dof - (int64_t)c->dir_dof.size();
    }
    GL_REQUIRE(b->E < ((int64_t)1 << 31), "batch too large for 32-bit element ids");
    b->d_parts.upload(b->parts, s);
    b->C.alloc(36 * b->E);
    b->geo.alloc(270 * b->E);
    b->f.alloc(b->N);
    std::vector<int64_t> hdir;
    std::vector<double> hval;
    for (int i = 0; i < n; ++i) {
        gl_ctx *c = b->items[i];
        const PartDesc &pd = b->parts[i];
        GL_CUDA(cudaMemcpyAsync(b->C.p + 36 * pd.elem_off, c->d_C.p, 36 * c->m.n_elem * sizeof(double),
                                cudaMemcpyDeviceToDevice, s));
        GL_CUDA(cudaMemcpyAsync(b->geo.p + 270 * pd.elem_off, c->d_geo.p, 270 * c->m.n_elem * sizeof(double),
                                cudaMemcpyDeviceToDevice, s));
        GL_CUDA(cudaMemcpyAsync(b->f.p + pd.dof_off, c->d_ftrac.p, c->m.n_dof * sizeof(double),
                                cudaMemcpyDeviceToDevice, s));
        for (size_t k = 0; k < c->dir_dof.size(); ++k) {
            hdir.push_back(c->dir_dof[k] + pd.dof_off);
            hval.push_back(c->dir_val[k]);
        }
    }
    b->ndir = (int64_t)hdir.size();
    b->d_dir.upload(hdir, s);
    b->d_dirval.upload(hval, s);
    // decomposition: given grid, or the autotuner per laminate
    b->grid.assign(n, {o.px, o.py});
    if (o.px <= 0 || o.py <= 0) {
        autotune_grids(b->items, is_dir, o.overlap, o.nev, o.precision == GL_PREC_MIXED, b->grid);
    }
    Problem &P = b->prob;
    P = Problem();
    P.stream = s;
    P.d_err = b->err.p;
    P.n_dof = b->N;
    P.n_elem = b->E;
    P.C = b->C.p;
    P.geo = b->geo.p;
    for (int i = 0; i < n; ++i) {
        const MeshHost &m = b->items[i]->m;
        const int px = std::min(b->grid[i][0], m.nx), py = std::min(b->grid[i][1], m.ny);
        b->grid[i] = {px, py};
        Part pt;
        pt.m = &m;
        pt.is_dir = std::move(is_dir[i]);
        pt.dof_off = b->parts[i].dof_off;
        pt.elem_off = b->parts[i].elem_off;
        pt.sub0 = (int)P.boxes.size();
        part_boxes(m, px, py, 1, o.overlap, P.boxes);
        pt.sub1 = (int)P.boxes.size();
        P.sub_part.resize(P.boxes.size(), i);
        P.parts.push_back(std::move(pt));
    }
    {
        std::vector<SubSymbolic> syms;
        problem_symbolic(P, false, LEAF_NODES, syms);
        build_plan(syms, b->PD, s);
        b->PD.ws_budget_bytes = b->opts.factor_ws_bytes > 0 ? b->opts.factor_ws_bytes : 6e9;
        b->PD.tc_update = b->opts.fp32_update == 0;
        b->PD.overlap_top = sweep_overlap_top(b->opts);
    }
    std::future<std::vector<SubSymbolic>> neumann;
    if (b->opts.nev > 0) neumann = neumann_symbolic(P, LEAF_NODES);
    if (b->opts.precision == GL_PREC_MIXED) {
        b->LD64.release();
        b->LD32.alloc(b->PD.l_size);
        numeric_factor<float>(b->PD, b->C.p, b->geo.p, nullptr, 0.0, b->LD32.p, b->err.p, s);
    } else {
        b->LD32.release();
        b->LD64.alloc(b->PD.l_size);
        numeric_factor<double>(b->PD, b->C.p, b->geo.p, nullptr, 0.0, b->LD64.p, b->err.p, s);
    }
    {
        int h = 0;
        GL_CUDA(cudaMemcpyAsync(&h, b->err.p, sizeof(int), cudaMemcpyDeviceToHost, s));
        GL_CUDA(cudaStreamSynchronize(s));
        if (h) {
            b->err.zero(s);
            if (h == 2) fail(GL_ERR_TIMEOUT, "batch local Dirichlet factorisation: a tensor-core wait gave up");
            fail(GL_ERR_NOT_SPD, "batch local Dirichlet factorisation: non-positive pivot");
        }
    }
    b->co = Coarse();
    if (b->opts.nev > 0) problem_coarse(P, b->opts, b->PD, neumann.get(), b->co);
    for (DBuf<double> *v : {&b->x, &b->r, &b->z, &b->p, &b->q, &b->ud, &b->fe}) v->alloc(b->N);
    b->c1.alloc(std::max(1, b->co.n0));
    b->c2.alloc(std::max(1, b->co.n0));
    if (b->opts.precision == GL_PREC_MIXED) b->xl32.alloc(3 * b->PD.n_local);
    else b->xl64.alloc(3 * b->PD.n_local);
    b->partials.alloc((size_t)n * SEG_BLOCKS);
    b->scal.alloc((size_t)6 * n);
    b->scal.zero(s);
    b->ints.alloc((size_t)2 * n + 1);
    b->ints.zero(s);
    if (!b->h_active) GL_CUDA(cudaMallocHost(&b->h_active, sizeof(int)));
    if (b->gexec) {
        cudaGraphExecDestroy(b->gexec);
        b->gexec = nullptr;
    }
    if (b->graph) {
        cudaGraphDestroy(b->graph);
        b->graph = nullptr;
    }
    GL_CUDA(cudaStreamSynchronize(s));
    b->ready = true;
    b->ms_setup = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
}

// One PCG iteration of every active laminate (captured once into a CUDA graph).
void batch_iteration(gl_batch *b) {
    cudaStream_t s = b->stream;
    const int n = (int)b->items.size();
    const int64_t N = b->N;
    SegScalars S = b->seg();
    batch_ku(b, b->p.p, b->q.p);
    set_entries(b->q.p, b->d_dir.p, b->ndir, nullptr, s);
    seg_dot(b->p.p, b->q.p, b->d_parts.p, n, b->partials.p, S.pq, s);
    seg_update_xr(b->x.p, b->r.p, b->p.p, b->q.p, b->d_parts.p, n, S, b->partials.p, s);
    seg_check(S, n, b->opts.tol, b->opts.max_iter, b->ints.p + 2 * n, s);
    if (b->opts.precision == GL_PREC_MIXED) seg_dot(b->r.p, b->z.p, b->d_parts.p, n, b->partials.p, S.rz_old, s);
    batch_precond(b, b->r.p, b->z.p);
    seg_dot(b->r.p, b->z.p, b->d_parts.p, n, b->partials.p, S.rho_new, s);
    seg_update_p(b->p.p, b->z.p, b->d_parts.p, n, S, s);
    (void)N;
}

void batch_solve(gl_batch *b, double *const *u, gl_info *infos) {
    if (!b->ready) fail(GL_ERR_STATE, "gl_batch_solve before gl_batch_setup");
    cudaStream_t s = b->stream;
    const int n = (int)b->items.size();
    const int64_t N = b->N;
    SegScalars S = b->seg();
    cudaEvent_t e0, e1;
    GL_CUDA(cudaEventCreate(&e0));
    GL_CUDA(cudaEventCreate(&e1));
    GL_CUDA(cudaEventRecord(e0, s));
    // fe = f - K u_D on the free DOFs
    b->ud.zero(s);
    set_entries(b->ud.p, b->d_dir.p, b->ndir, b->d_dirval.p, s);
    batch_ku(b, b->ud.p, b->q.p);
    sub(b->fe.p, b->f.p, b->q.p, N, s);
    set_entries(b->fe.p, b->d_dir.p, b->ndir, nullptr, s);
    seg_dot(b->fe.p, b->fe.p, b->d_parts.p, n, b->partials.p, S.ff, s);
    k_seg_init<<<(n + 127) / 128, 128, 0, s>>>(S, n);
    b->x.zero(s);
    GL_CUDA(cudaMemcpyAsync(b->r.p, b->fe.p, N * sizeof(double), cudaMemcpyDeviceToDevice, s));
    batch_precond(b, b->r.p, b->z.p);
    seg_dot(b->r.p, b->z.p, b->d_parts.p, n, b->partials.p, S.rho, s);
    GL_CUDA(cudaMemcpyAsync(b->p.p, b->z.p, N * sizeof(double), cudaMemcpyDeviceToDevice, s));
    g_launches += 2 * (b->ndir ? 1 : 0) + 6;
    if (!b->gexec) {
        GL_CUDA(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
        const long long before = g_launches.load();
        batch_iteration(b);
        g_launches.store(before);   // counted per replay below
        GL_CUDA(cudaStreamEndCapture(s, &b->graph));
        GL_CUDA(cudaGraphInstantiate(&b->gexec, b->graph, 0));
    }
    const int per_iter = 6 + (b->ndir ? 1 : 0) + (b->opts.precision == GL_PREC_MIXED ? 2 : 0) + 2 +
                         (int)factor_solve_launches(b->PD) + (b->co.n0 > 0 ? 3 : 0) + 4;
    const int period = b->opts.resid_period;
    for (int it = 1; it <= b->opts.max_iter; ++it) {
        GL_CUDA(cudaGraphLaunch(b->gexec, s));
        g_launches += per_iter;
        GL_CUDA(cudaMemcpyAsync(b->h_active, b->ints.p + 2 * n, sizeof(int), cudaMemcpyDeviceToHost, s));
        GL_CUDA(cudaStreamSynchronize(s));
        if (*b->h_active == 0) {
            if (b->opts.precision != GL_PREC_MIXED) break;
            // mixed: every laminate stopped on its recurrence residual; confirm on the FP64 true
            // residual r = fe - K x and restart (z = M r, p = z) those that miss tol
            batch_ku(b, b->x.p, b->q.p);
            set_entries(b->q.p, b->d_dir.p, b->ndir, nullptr, s);
            sub(b->r.p, b->fe.p, b->q.p, N, s);
            seg_dot(b->r.p, b->r.p, b->d_parts.p, n, b->partials.p, S.rr, s);
            seg_confirm(S, n, b->opts.tol, b->opts.max_iter, b->ints.p + 2 * n, s);
            g_launches += 4 + (b->ndir ? 1 : 0);
            GL_CUDA(cudaMemcpyAsync(b->h_active, b->ints.p + 2 * n, sizeof(int), cudaMemcpyDeviceToHost, s));
            GL_CUDA(cudaStreamSynchronize(s));
            if (*b->h_active == 0) break;
            batch_precond(b, b->r.p, b->z.p);
            seg_dot(b->r.p, b->z.p, b->d_parts.p, n, b->partials.p, S.rho, s);
            GL_CUDA(cudaMemcpyAsync(b->p.p, b->z.p, N * sizeof(double), cudaMemcpyDeviceToDevice, s));
            g_launches += 2;
            continue;
        }
        if (b->opts.precision == GL_PREC_MIXED && it % period == 0) {
            // FP64 residual replacement r = fe - K x (frozen laminates keep their r: x is unchanged)
            batch_ku(b, b->x.p, b->q.p);
            set_entries(b->q.p, b->d_dir.p, b->ndir, nullptr, s);
            sub(b->r.p, b->fe.p, b->q.p, N, s);
            g_launches += 2 + (b->ndir ? 1 : 0);
        }
    }
    // results: recurrence residuals, FP64 true residuals, displacements
    std::vector<double> hs((size_t)6 * n);
    std::vector<int> hi((size_t)2 * n);
    GL_CUDA(cudaMemcpyAsync(hs.data(), b->scal.p, hs.size() * sizeof(double), cudaMemcpyDeviceToHost, s));
    GL_CUDA(cudaMemcpyAsync(hi.data(), b->ints.p, hi.size() * sizeof(int), cudaMemcpyDeviceToHost, s));
    batch_ku(b, b->x.p, b->q.p);
    set_entries(b->q.p, b->d_dir.p, b->ndir, nullptr, s);
    sub(b->r.p, b->fe.p, b->q.p, N, s);
    seg_dot(b->r.p, b->r.p, b->d_parts.p, n, b->partials.p, S.rr, s);
    axpy(b->x.p, 1.0, b->ud.p, N, s);
    g_launches += 6;
    std::vector<double> hrt(n);
    GL_CUDA(cudaMemcpyAsync(hrt.data(), S.rr, n * sizeof(double), cudaMemcpyDeviceToHost, s));
    GL_CUDA(cudaEventRecord(e1, s));
    GL_CUDA(cudaStreamSynchronize(s));
    float ms = 0;
    GL_CUDA(cudaEventElapsedTime(&ms, e0, e1));
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    int worst = GL_OK;
    for (int i = 0; i < n; ++i) {
        const double ff = hs[4 * n + i], rr = hs[3 * n + i];
        const int iters = hi[n + i];
        int st = GL_OK;
        // mixed: accepted on the FP64 true residual; FP64: on the recurrence residual
        const double racc = b->opts.precision == GL_PREC_MIXED ? hrt[i] : rr;
        if (!std::isfinite(rr) || !std::isfinite(racc)) st = GL_ERR_NAN;
        else if (ff > 0 && racc > b->opts.tol * b->opts.tol * ff) st = GL_ERR_NOT_CONVERGED;
        if (st != GL_OK) worst = st;
        if (u[i]) from_device(u[i], b->x.p + b->parts[i].dof_off, b->parts[i].n_dof, s);
        if (infos) {
            gl_info &in = infos[i];
            in.iters = iters;
            in.status = st;
            in.rel_resid = ff > 0 ? std::sqrt(rr / ff) : 0.0;
            in.rel_resid_true = ff > 0 ? std::sqrt(hrt[i] / ff) : 0.0;
            in.ms_setup = b->ms_setup;
            in.ms_solve = ms;
            in.n_free = b->n_free[i];
            in.n_coarse = (int)(b->co.n0 ? b->co.kn[i] : 0);
            in.n_coarse_dropped = b->co.part_dropped.empty() ? 0 : b->co.part_dropped[i];
            in.factor_nnz = b->PD.l_size;
        }
    }
    if (worst != GL_OK) {
        g_last_error = worst == GL_ERR_NAN ? "NaN/Inf in a batched PCG iteration" : "a laminate reached max_iter";
        throw Error{worst, g_last_error};
    }
}

}  // namespace

// ====================================================================== C ABI

extern "C" {

const char *gl_strerror(int code) {
    switch (code) {
        case GL_OK: return "ok";
        case GL_ERR_INVALID_ARG: return "invalid argument";
        case GL_ERR_OOM: return "out of memory";
        case GL_ERR_CUDA: return "CUDA error";
        case GL_ERR_NOT_SPD: return "matrix not positive definite";
        case GL_ERR_NOT_CONVERGED: return "not converged";
        case GL_ERR_NAN: return "NaN or Inf";
        case GL_ERR_TIMEOUT: return "device wait timed out";
        case GL_ERR_STATE: return "call out of order";
        default: return "unknown error";
    }
}

const char *gl_last_error(void) { return g_last_error.c_str(); }

int gl_create(gl_ctx **out, int device, void *cuda_stream) {
    return guard([&] {
        GL_REQUIRE(out, "null output pointer");
        int n = 0;
        GL_CUDA(cudaGetDeviceCount(&n));
        GL_REQUIRE(device >= 0 && device < n, "no such CUDA device");
        GL_CUDA(cudaSetDevice(device));
        gl_ctx *c = new gl_ctx();
        c->device = device;
        c->stream = (cudaStream_t)cuda_stream;
        *out = c;
    });
}

void gl_destroy(gl_ctx *ctx) {
    if (!ctx) return;
    cudaSetDevice(ctx->device);
    cudaStreamSynchronize(ctx->stream);
    delete ctx;
}

int gl_set_materials(gl_ctx *c, int n_ortho, const gl_ortho *ortho, int n_iso, const double *E_nu) {
    return guard([&] {
        require_ctx(c);
        GL_REQUIRE(n_ortho >= 0 && n_iso >= 0 && n_ortho + n_iso > 0, "empty material table");
        auto ho = fetch(ortho, n_ortho);
        auto hi = fetch(E_nu, 2 * (size_t)n_iso);
        c->matC.clear();
        c->mat_iso.clear();
        for (auto &o : ho) {
            GL_REQUIRE(o.E1 > 0 && o.E2 > 0 && o.E3 > 0 && o.G12 > 0 && o.G13 > 0 && o.G23 > 0,
                       "orthotropic moduli must be positive");
            double S[36] = {0};
            S[0] = 1 / o.E1; S[7] = 1 / o.E2; S[14] = 1 / o.E3;
            S[1] = S[6] = -o.nu12 / o.E1;
            S[2] = S[12] = -o.nu13 / o.E1;
            S[8] = S[13] = -o.nu23 / o.E2;
            S[21] = 1 / o.G23; S[28] = 1 / o.G13; S[35] = 1 / o.G12;
            double C[36];
            inv6(S, C);
            c->matC.insert(c->matC.end(), C, C + 36);
            c->mat_iso.push_back(0);
        }
        for (int i = 0; i < n_iso; ++i) {
            double E = hi[2 * i], nu = hi[2 * i + 1];
            GL_REQUIRE(E > 0 && nu > -1 && nu < 0.5, "isotropic constants out of range");
            double lam = E * nu / ((1 + nu) * (1 - 2 * nu)), mu = E / (2 * (1 + nu));
            double C[36] = {0};
            for (int a = 0; a < 3; ++a)
                for (int b = 0; b < 3; ++b) C[6 * a + b] = lam + (a == b ? 2 * mu : 0);
            C[21] = C[28] = C[35] = mu;
            c->matC.insert(c->matC.end(), C, C + 36);
            c->mat_iso.push_back(1);
        }
        c->have_mat = true;
        c->ready = false;
    });
}

int gl_set_mesh(gl_ctx *c, const gl_mesh *mesh) {
    return guard([&] {
        require_ctx(c);
        GL_REQUIRE(mesh, "null mesh");
        GL_REQUIRE(c->have_mat, "gl_set_materials must come before gl_set_mesh");
        GL_REQUIRE(mesh->nx >= 1 && mesh->ny >= 1 && mesh->nlayers >= 1, "empty mesh");
        GL_REQUIRE(mesh->geometry == 0 || mesh->geometry == 1, "geometry must be 0 or 1");
        GL_REQUIRE(mesh->element == 0 || mesh->element == 1, "element must be 0 (Q2) or 1 (serendipity)");
        GL_REQUIRE(mesh->periodic_width == 0 || mesh->periodic_width == 1, "periodic_width must be 0 or 1");
        GL_REQUIRE(!mesh->periodic_width || (mesh->element == 0 && mesh->ny >= 2),
                   "periodic width needs the Q2 element and at least 2 elements across the width");
        MeshHost m;
        m.nx = mesh->nx;
        m.ny = mesh->ny;
        m.sv = fetch(mesh->x, m.nx + 1);
        m.lv = fetch(mesh->y, m.ny + 1);
        auto nel = fetch(mesh->layer_nel, mesh->nlayers);
        auto th = fetch(mesh->layer_thick, mesh->nlayers);
        m.layer_mat = fetch(mesh->layer_mat, mesh->nlayers);
        auto ang = fetch(mesh->layer_angle_deg, mesh->nlayers);
        for (int i = 0; i < m.nx; ++i) GL_REQUIRE(m.sv[i + 1] > m.sv[i], "x vertices must increase");
        for (int i = 0; i < m.ny; ++i) GL_REQUIRE(m.lv[i + 1] > m.lv[i], "y vertices must increase");
        m.rv.assign(1, 0.0);
        double base = 0.0;
        for (int k = 0; k < mesh->nlayers; ++k) {
            GL_REQUIRE(nel[k] >= 1 && th[k] > 0, "layers need >= 1 element and positive thickness");
            GL_REQUIRE(m.layer_mat[k] >= 0 && m.layer_mat[k] < (int)c->mat_iso.size(), "layer material out of range");
            for (int i = 0; i < nel[k]; ++i) {
                m.rv.push_back(base + th[k] * (i + 1) / nel[k]);
                m.layer_of_ez.push_back(k);
            }
            base += th[k];
            m.layer_angle.push_back(ang[k] * M_PI / 180.0);
        }
        m.nz = (int)m.layer_of_ez.size();
        m.NX = 2 * m.nx + 1;
        m.NY = 2 * m.ny + 1;
        m.NZ = 2 * m.nz + 1;
        m.n_nodes = (int64_t)m.NX * m.NY * m.NZ;
        m.n_dof = 3 * m.n_nodes;
        m.n_elem = (int64_t)m.nx * m.ny * m.nz;
        GL_REQUIRE(m.n_dof < (int64_t)1 << 31, "mesh too large for 32-bit local indices");
        m.geometry = mesh->geometry;
        m.element = mesh->element;
        m.periodic = mesh->periodic_width != 0;
        m.R_inner = mesh->R_inner;
        m.limb_L = mesh->limb_L;
        m.arc_rad = mesh->arc_deg * M_PI / 180.0;
        if (m.geometry == 1) GL_REQUIRE(m.R_inner > 0 && m.arc_rad > 0, "curved mesh needs R_inner > 0, arc > 0");
        auto mid = [](const std::vector<double> &v) {
            std::vector<double> o(2 * v.size() - 1);
            for (size_t i = 0; i < v.size(); ++i) o[2 * i] = v[i];
            for (size_t i = 0; i + 1 < v.size(); ++i) o[2 * i + 1] = 0.5 * (v[i] + v[i + 1]);
            return o;
        };
        m.tn = mid(m.sv);
        m.ln = mid(m.lv);
        m.rn = mid(m.rv);
        if (mesh->theta_e) m.theta = fetch(mesh->theta_e, m.n_elem);
        if (mesh->elem_mat) {
            m.elem_mat = fetch(mesh->elem_mat, m.n_elem);
            for (int v : m.elem_mat)
                GL_REQUIRE(v >= 0 && v < (int)c->mat_iso.size(), "element material out of range");
        }
        if (mesh->node_dr) {
            m.node_dr = fetch(mesh->node_dr, m.n_nodes);
            // every through-thickness node column must stay strictly increasing
            for (int64_t col = 0; col < (int64_t)m.NX * m.NY; ++col)
                for (int iz = 0; iz + 1 < m.NZ; ++iz) {
                    const int64_t a = col + (int64_t)m.NX * m.NY * iz, b = a + (int64_t)m.NX * m.NY;
                    GL_REQUIRE(std::isfinite(m.node_dr[a]) && std::isfinite(m.node_dr[b]) &&
                                   m.rn[iz] + m.node_dr[a] < m.rn[iz + 1] + m.node_dr[b],
                               "node_dr folds a through-thickness node column");
                }
        }
        c->m = std::move(m);
        c->have_mesh = true;
        c->ready = false;
        c->dir_dof.clear();
        c->dir_val.clear();
        c->tractions.clear();
    });
}

int gl_set_dirichlet(gl_ctx *c, int64_t n, const int64_t *dof, const double *val) {
    return guard([&] {
        require_ctx(c);
        GL_REQUIRE(c->have_mesh, "gl_set_mesh must come first");
        GL_REQUIRE(n >= 0, "negative count");
        auto d = fetch(dof, n);
        auto v = fetch(val, n);
        std::vector<std::pair<int64_t, double>> pv;
        for (int64_t i = 0; i < n; ++i) {
            GL_REQUIRE(d[i] >= 0 && d[i] < c->m.n_dof, "Dirichlet DOF out of range");
            pv.push_back({d[i], v[i]});
        }
        std::sort(pv.begin(), pv.end());
        c->dir_dof.clear();
        c->dir_val.clear();
        for (auto &q : pv) {
            if (!c->dir_dof.empty() && c->dir_dof.back() == q.first) {
                c->dir_val.back() = q.second;
                continue;
            }
            c->dir_dof.push_back(q.first);
            c->dir_val.push_back(q.second);
        }
        c->d_dir_dof.upload(c->dir_dof, c->stream);
        c->d_dir_val.upload(c->dir_val, c->stream);
        GL_CUDA(cudaStreamSynchronize(c->stream));
        c->ready = false;
    });
}

int gl_set_traction(gl_ctx *c, int face, const double t[3]) {
    return guard([&] {
        require_ctx(c);
        GL_REQUIRE(c->have_mesh, "gl_set_mesh must come first");
        GL_REQUIRE(face >= 0 && face < 6, "face must be in 0..5");
        auto h = fetch(t, 3);
        c->tractions.push_back({face, {h[0], h[1], h[2]}});
        c->ready = false;
    });
}

int gl_setup(gl_ctx *c, const gl_opts *o) {
    return guard([&] {
        require_ctx(c);
        GL_REQUIRE(o, "null options");
        setup(c, *o);
    });
}

int gl_num_dofs(const gl_ctx *c, int64_t *n) {
    return guard([&] {
        GL_REQUIRE(c && n && c->have_mesh, "no mesh");
        *n = c->m.n_dof;
    });
}

int gl_num_elems(const gl_ctx *c, int64_t *n) {
    return guard([&] {
        GL_REQUIRE(c && n && c->have_mesh, "no mesh");
        *n = c->m.n_elem;
    });
}

int gl_rhs(gl_ctx *c, double *f) {
    return guard([&] {
        require_ctx(c);
        if (!c->ready) fail(GL_ERR_STATE, "gl_rhs before gl_setup");
        GL_REQUIRE(f, "null output");
        from_device(f, c->d_ftrac.p, c->m.n_dof, c->stream);
    });
}

int gl_solve(gl_ctx *c, const double *f, double *u, gl_info *info) {
    return guard([&] {
        require_ctx(c);
        GL_REQUIRE(u, "null output");
        solve(c, f, u, info);
    });
}

int gl_solve_increment(gl_ctx *c, const double *g, double *du, gl_info *info) {
    return guard([&] {
        require_ctx(c);
        GL_REQUIRE(g && du, "null argument");
        solve(c, g, du, info, true);                 // K_ff du_f = g_f, du = 0 on Dirichlet DOFs
    });
}

int gl_stress(gl_ctx *c, const double *u, double *s33, double *t13, double *peak) {
    return guard([&] {
        require_ctx(c);
        if (!c->ready) fail(GL_ERR_STATE, "gl_stress before gl_setup");
        GL_REQUIRE(u, "null displacement");
        cudaStream_t s = c->stream;
        const MeshHost &m = c->m;
        // outputs in host memory (or over u) go through the work vectors z and r
        const double *du = field_in(c, u);
        auto out = [&](double *p, DBuf<double> &w, const double *peer) {
            return in_place(c, {p, m.n_elem}, {{u, m.n_dof}, {peer, m.n_elem}}) ? p : w.p;
        };
        double *d33 = out(s33, c->z, t13), *d13 = out(t13, c->r, s33);
        launch_stress(m, c->d_X.p, c->d_C.p, c->d_psi.p, du, d33, d13, s);
        g_launches += 1 + (peak ? 2 : 0);
        if (peak) {
            max_where(d33, c->d_resin.p, m.n_elem, c->partials.p, &c->S.p->alpha, s);
            GL_CUDA(cudaMemcpyAsync(c->h_pin, &c->S.p->alpha, sizeof(double), cudaMemcpyDeviceToHost, s));
        }
        if (s33 && s33 != d33) to_device(s33, d33, m.n_elem, s);
        if (t13 && t13 != d13) to_device(t13, d13, m.n_elem, s);
        finish_scalar(c, peak, &c->S.p->alpha, c->h_pin);
    });
}

int gl_stress_noalloc(gl_ctx *c, const double *u, double *s33, double *t13, double *peak) {
    return guard([&] {
        require_ctx(c);
        if (!c->ready) fail(GL_ERR_STATE, "gl_stress_noalloc before gl_setup");
        GL_REQUIRE(u && s33 && t13, "gl_stress_noalloc: u, s33 and t13 are required");
        auto on_ctx_device = [&](const void *p) {
            cudaPointerAttributes a{};
            if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
                cudaGetLastError();
                return false;
            }
            return (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged) && a.device == c->device;
        };
        // each buffer in turn: device memory of the context's device, long enough for what the
        // kernels touch (N doubles of u read; n_elem doubles of s33, t13 and one of peak written);
        // all checks come before the first launch
        auto check = [&](const void *p, size_t bytes, const char *name) {
            GL_REQUIRE(on_ctx_device(p), std::string("gl_stress_noalloc: ") + name +
                                             " must be device memory of the context's device");
            require_device_span(p, bytes, (std::string("gl_stress_noalloc: ") + name).c_str());
        };
        check(u, c->m.n_dof * sizeof(double), "u");
        check(s33, c->m.n_elem * sizeof(double), "s33");
        check(t13, c->m.n_elem * sizeof(double), "t13");
        if (peak) check(peak, sizeof(double), "peak_s33");
        stress_noalloc(c->m, c->device, c->d_X.p, c->d_C.p, c->d_psi.p, c->d_resin.p, u, s33, t13, peak, c->stream);
        g_launches += 1 + (peak ? 2 : 0);
    });
}

int gl_apply_K(gl_ctx *c, const double *x, double *y) {
    return guard([&] {
        require_ctx(c);
        if (!c->ready) fail(GL_ERR_STATE, "gl_apply_K before gl_setup");
        GL_REQUIRE(x && y, "null vector");
        cudaStream_t s = c->stream;
        const int64_t N = c->m.n_dof;
        const double *dx = x;
        if (!in_place(c, {x, N})) {
            to_device(c->p.p, x, N, s);
            dx = c->p.p;
        }
        double *dy = in_place(c, {y, N}, {{x, N}}) ? y : c->q.p;
        apply_K(c, dx, dy);
        if (dy != y) to_device(y, dy, N, s);
        GL_CUDA(cudaStreamSynchronize(s));
    });
}

int gl_apply_prec(gl_ctx *c, const double *r, double *z) {
    return guard([&] {
        require_ctx(c);
        if (!c->ready) fail(GL_ERR_STATE, "gl_apply_prec before gl_setup");
        GL_REQUIRE(r && z, "null vector");
        cudaStream_t s = c->stream;
        to_device(c->r.p, r, c->m.n_dof, s);
        set_entries(c->r.p, c->d_dir_dof.p, c->n_dir, nullptr, s);
        apply_prec(c, c->r.p, c->z.p);
        from_device(z, c->z.p, c->m.n_dof, s);
    });
}

int gl_failure_index(gl_ctx *c, const double *u, double s33_allow, double s13_allow, double *F, double *peak,
                     int64_t *peak_elem) {
    return guard([&] {
        require_ctx(c);
        if (!c->ready) fail(GL_ERR_STATE, "gl_failure_index before gl_setup");
        GL_REQUIRE(u, "null displacement");
        GL_REQUIRE(s33_allow > 0 && s13_allow > 0, "allowables must be positive");
        const MeshHost &m = c->m;
        GL_REQUIRE(m.n_elem < (int64_t)1 << 24, "gl_failure_index: at most 16,777,215 elements");
        cudaStream_t s = c->stream;
        const double *du = field_in(c, u);
        double *dF = in_place(c, {F, m.n_elem}, {{u, m.n_dof}}) ? F : c->z.p;
        launch_failure(m, c->d_X.p, c->d_C.p, c->d_psi.p, c->d_resin.p, du, s33_allow, s13_allow, dF, c->partials.p, s);
        g_launches += 2;
        GL_CUDA(cudaMemcpyAsync(c->h_pin, c->partials.p, 2 * sizeof(double), cudaMemcpyDeviceToHost, s));
        if (F && F != dF) to_device(F, dF, m.n_elem, s);
        finish_scalar(c, peak, c->partials.p + 1, c->h_pin + 1);
        int64_t key;
        std::memcpy(&key, c->h_pin, sizeof(key));
        if (peak_elem) *peak_elem = key & 0xFFFFFF;
    });
}

int gl_set_theta(gl_ctx *c, const double *theta_e) {
    return guard([&] {
        require_ctx(c);
        GL_REQUIRE(c->have_mesh, "gl_set_mesh must come first");
        GL_REQUIRE(theta_e, "null theta");
        MeshHost &m = c->m;
        m.theta = fetch(theta_e, m.n_elem);
        if (c->ready) {
            // new C_e for K u and the stresses; the factors and the coarse space are kept
            c->d_theta.upload(m.theta, c->stream);
            launch_elem_material(m.n_elem, m.nx, m.ny, c->d_layer_of_ez.p, c->d_layer_mat.p, c->d_elem_mat.p,
                                 c->d_layer_angle.p, c->d_theta.p, c->d_psi.p, c->d_matC.p, c->d_C.p, c->stream);
            GL_CUDA(cudaStreamSynchronize(c->stream));
        }
    });
}

int gl_stress_vjp(gl_ctx *c, const double *u, const double *w33, const double *w13, double *dJdu, double *dJdth) {
    return guard([&] {
        require_ctx(c);
        if (!c->ready) fail(GL_ERR_STATE, "gl_stress_vjp before gl_setup");
        GL_REQUIRE(u, "null displacement");
        cudaStream_t s = c->stream;
        const MeshHost &m = c->m;
        const int64_t N = m.n_dof, E = m.n_elem;
        const double *du = field_in(c, u);
        auto weights = [&](const double *w, DBuf<double> &stage) -> const double * {
            if (!w || in_place(c, {w, E})) return w;
            to_device(stage.p, w, E, s);
            return stage.p;
        };
        const double *d33 = weights(w33, c->z), *d13 = weights(w13, c->r);
        const Span in[3] = {{u, N}, {w33, E}, {w13, E}};
        double *dgu = !dJdu ? nullptr : (in_place(c, {dJdu, N}, {in[0], in[1], in[2]}) ? dJdu : c->p.p);
        double *dgt = !dJdth ? nullptr
                             : (in_place(c, {dJdth, E}, {in[0], in[1], in[2], {dJdu, N}}) ? dJdth : c->fe.p);
        if (dgu) GL_CUDA(cudaMemsetAsync(dgu, 0, N * sizeof(double), s));
        launch_stress_vjp(m, c->d_X.p, c->d_C.p, c->d_psi.p, c->d_layer_of_ez.p, c->d_layer_mat.p, c->d_elem_mat.p,
                          c->d_layer_angle.p, c->d_theta.p, c->d_matC.p, du, d33, d13, dgu, dgt, s);
        g_launches += 1;
        if (dgu && has_slaves(m)) slave_fold(m, dgu, s);   // dJ/du = P^T dJ/du_Q2
        if (dgu && dgu != dJdu) to_device(dJdu, dgu, N, s);
        if (dgt && dgt != dJdth) to_device(dJdth, dgt, E, s);
        GL_CUDA(cudaStreamSynchronize(s));
    });
}

int gl_adjoint(gl_ctx *c, const double *u, const double *dJdu, double *grad, gl_info *info) {
    return guard([&] {
        require_ctx(c);
        if (!c->ready) fail(GL_ERR_STATE, "gl_adjoint before gl_setup");
        GL_REQUIRE(u && dJdu && grad, "null argument");
        cudaStream_t s = c->stream;
        const MeshHost &m = c->m;
        solve(c, dJdu, c->x.p, info, true);          // K_ff lambda = (dJ/du)_f, lambda = 0 on Dirichlet DOFs
        const double *du = field_in(c, u);           // lambda comes back filled from solve()
        double *dg = in_place(c, {grad, m.n_elem}, {{u, m.n_dof}}) ? grad : c->z.p;
        launch_adjoint_contract(m, c->d_geo.p, c->d_layer_of_ez.p, c->d_layer_mat.p, c->d_elem_mat.p,
                                c->d_layer_angle.p,
                                c->d_theta.p, c->d_psi.p, c->d_matC.p, du, c->x.p, dg, s);
        g_launches += 1;
        if (dg != grad) to_device(grad, dg, m.n_elem, s);
        GL_CUDA(cudaStreamSynchronize(s));
    });
}

int gl_profile(gl_ctx *c, int enable) {
    return guard([&] {
        require_ctx(c);
        Prof &P = c->prof;
        if (enable && !P.on)
            for (auto &e : P.ev) GL_CUDA(cudaEventCreate(&e));
        if (!enable && P.on) {
            GL_CUDA(cudaStreamSynchronize(c->stream));
            for (auto &e : P.ev) cudaEventDestroy(e);
        }
        GL_REQUIRE(enable >= 0 && enable <= 2, "gl_profile: enable must be 0, 1 or 2");
        P.on = enable != 0;
        P.levels = enable == 2;
        if (c->ready) level_clock_enable(c->PD, P.levels);
        for (int i = 0; i < PH_N; ++i) {
            P.ms[i] = 0;
            P.count[i] = 0;
            P.pending[i] = 0;
        }
    });
}

int gl_profile_read(gl_ctx *c, gl_profile_data *out) {
    return guard([&] {
        require_ctx(c);
        GL_REQUIRE(out, "null output");
        for (int ph = 0; ph < PH_N; ++ph) prof_fold(c, ph);
        out->ms_ku = c->prof.ms[PH_KU];
        out->ms_local = c->prof.ms[PH_LOCAL];
        out->ms_coarse = c->prof.ms[PH_COARSE];
        out->n_ku = c->prof.count[PH_KU];
        out->n_local = c->prof.count[PH_LOCAL];
        out->n_coarse = c->prof.count[PH_COARSE];
        out->factor_entries = c->PD.l_size;
        out->factor_nonzeros = c->PD.nnz;
        out->local_dofs = c->PD.n_local;
        out->factor_bytes_per_entry = c->opts.precision == GL_PREC_MIXED ? 4 : 8;
        out->n_elem = c->m.n_elem;
        out->n_dof = c->m.n_dof;
        out->n_sub = (int)c->prob.boxes.size();
        out->n_coarse_dim = c->co.n0;
        out->factor_levels = 0;
        out->max_level_fronts = 0;
        for (auto &L : c->PD.levels) {
            if (!L.fronts.empty()) ++out->factor_levels;
            out->max_level_fronts = std::max(out->max_level_fronts, (int)L.fronts.size());
        }
        out->factor_groups = c->PD.last_groups;
        out->eig_groups = c->co.n_groups;
    });
}

int gl_profile_levels(gl_ctx *c, int max_levels, double *fwd_ms, double *bwd_ms, int64_t *fronts,
                      int64_t *nonzeros, int64_t *padded, int *max_front, int *n_levels, int64_t *calls) {
    return guard([&] {
        require_ctx(c);
        if (!c->ready) fail(GL_ERR_STATE, "gl_profile_levels before gl_setup");
        GL_REQUIRE(max_levels >= 0, "max_levels must be >= 0");
        const FactorPlan &P = c->PD;
        const int nlev = (int)P.levels.size();
        if (n_levels) *n_levels = nlev;
        if (calls) *calls = P.clock.calls;
        for (int d = 0; d < std::min(nlev, max_levels); ++d) {
            const Level &Lv = P.levels[d];
            int64_t nz = 0, pad = 0;
            for (int g : Lv.fronts) {
                const FrontDesc &fd = P.fr[g];
                nz += (int64_t)fd.p * (fd.p + 1) / 2 + (int64_t)fd.p * fd.q;
                for (int jb = 0; jb < fd.p; jb += 32) pad += 32 * (int64_t)(fd.p + fd.q - jb);
            }
            const bool have = d < (int)P.clock.fwd_ms.size();
            if (fwd_ms) fwd_ms[d] = have ? P.clock.fwd_ms[d] : 0.0;
            if (bwd_ms) bwd_ms[d] = have ? P.clock.bwd_ms[d] : 0.0;
            if (fronts) fronts[d] = (int64_t)Lv.fronts.size();
            if (nonzeros) nonzeros[d] = nz;
            if (padded) padded[d] = pad;
            if (max_front) max_front[d] = Lv.max_f;
        }
    });
}

long long gl_kernel_launches(void) { return g_launches.load(); }

int gl_fp64_peak_probe(int device, int iters, int reps, double *flops_per_s, int *n_sm, double *ms) {
    return guard([&] {
        GL_REQUIRE(flops_per_s, "null output");
        GL_REQUIRE(iters > 0 && reps > 0, "iters and reps must be positive");
        int ndev = 0;
        GL_CUDA(cudaGetDeviceCount(&ndev));
        GL_REQUIRE(device >= 0 && device < ndev, "no such device");
        GL_CUDA(cudaSetDevice(device));
        *flops_per_s = fp64_probe(iters, reps, n_sm, ms);
    });
}

int gl_geneo_eigenvalues(gl_ctx *c, double *lambda, int capacity, int *count) {
    return guard([&] {
        require_ctx(c);
        if (!c->ready) fail(GL_ERR_STATE, "before gl_setup");
        GL_REQUIRE(count, "null count");
        *count = (int)c->co.eig.size();
        if (lambda) {
            GL_REQUIRE(capacity >= (int)c->co.eig.size(), "capacity too small");
            std::copy(c->co.eig.begin(), c->co.eig.end(), lambda);
        }
    });
}

int gl_batch_create(gl_batch **out, int n, gl_ctx *const *items, void *cuda_stream) {
    return guard([&] {
        GL_REQUIRE(out && n >= 1 && items, "need at least one laminate");
        gl_batch *b = new gl_batch();
        try {
            b->device = items[0]->device;
            for (int i = 0; i < n; ++i) {
                GL_REQUIRE(items[i], "null laminate");
                GL_REQUIRE(items[i]->device == b->device, "all laminates of a batch must be on one device");
                GL_REQUIRE(!items[i]->have_mesh || (items[i]->m.element == 0 && !items[i]->m.periodic),
                           "the batched engine takes Q2 laminates without periodic width conditions only");
                for (int j = 0; j < i; ++j) GL_REQUIRE(items[j] != items[i], "a laminate appears twice in the batch");
                b->items.push_back(items[i]);
                b->item_streams.push_back(items[i]->stream);
            }
            GL_CUDA(cudaSetDevice(b->device));
            if (cuda_stream) {
                b->stream = (cudaStream_t)cuda_stream;
            } else {
                GL_CUDA(cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking));
                b->own_stream = true;
            }
        } catch (...) {
            delete b;
            throw;
        }
        *out = b;
    });
}

int gl_batch_setup(gl_batch *b, const gl_opts *opts) {
    return guard([&] {
        GL_REQUIRE(b && opts, "null argument");
        GL_CUDA(cudaSetDevice(b->device));
        batch_setup(b, *opts);
    });
}

int gl_batch_solve(gl_batch *b, double *const *u, gl_info *infos) {
    return guard([&] {
        GL_REQUIRE(b && u, "null argument");
        GL_CUDA(cudaSetDevice(b->device));
        batch_solve(b, u, infos);
    });
}

int gl_batch_grid(const gl_batch *b, int *pxpy) {
    return guard([&] {
        GL_REQUIRE(b && pxpy && b->ready, "batch not set up");
        for (size_t i = 0; i < b->grid.size(); ++i) {
            pxpy[2 * i] = b->grid[i][0];
            pxpy[2 * i + 1] = b->grid[i][1];
        }
    });
}

void gl_batch_destroy(gl_batch *b) {
    if (!b) return;
    cudaSetDevice(b->device);
    cudaStreamSynchronize(b->stream);
    delete b;
}

}  // extern "C"
