// C ABI of the library (include/rich.h): owns the device memory of a
// simulation, builds its first mesh on the host (a0), and enqueues the device
// sweep (a1-a9) and the mesh's update for the moved points (a0) on CUDA
// streams.  There is no CPU fallback: without a CUDA device rich_init_mesh
// fails with RICH_ENODEV.
#include <array>
#include <chrono>
#include <climits>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <memory>
#include <new>
#include <string>
#include <thread>
#include <vector>

#include <cuda_runtime.h>

#include "../../include/rich.h"
#include "api_internal.h"
#include "mesh.h"
#include "meshupdate.h"
#include "meshupdate_dev.h"
#include "sweep.cuh"
#include "threadpool.h"

namespace rich {
namespace {
thread_local std::string g_last_error;
}
int set_error(int code, const std::string &msg)
{
    g_last_error = msg;
    return code;
}
const char *last_error() { return g_last_error.c_str(); }
}  // namespace rich

namespace {

using rich::DBuf;
using rich::now_ms;
using rich::upload;
#define CUDA_TRY RICH_CUDA_TRY

int fail(int code, const std::string &msg) { return rich::set_error(code, msg); }

int mesh_rc(int rc)
{
    switch (rc) {
    case 0: return RICH_OK;
    case -2: return fail(RICH_EDUPLICATE, "two generating points coincide");
    case -4: return fail(RICH_ETOOFEW, "too few points: the ghost band cannot close every cell");
    default: return fail(RICH_ETESS, "tessellation failed");
    }
}

}  // namespace

namespace rich {
bool valid_config(const rich_config *c)
{
    return c && c->gamma > 1.0 && std::isfinite(c->gamma) && c->cfl > 0.0 && c->x1 > c->x0 && c->y1 > c->y0 &&
           (c->boundary == RICH_BC_REFLECTIVE || c->boundary == RICH_BC_PERIODIC) &&
           (c->motion == RICH_MESH_LAGRANGIAN || c->motion == RICH_MESH_EULERIAN) && c->limiter >= 0 &&
           c->limiter <= 2 && (c->scheme == RICH_SCHEME_EXTRAPOLATED || c->scheme == RICH_SCHEME_TIME_CENTRED) && (c->precision == RICH_FP64 || c->precision == RICH_FP32_SPLIT) && c->chi >= 0 &&
           c->eta >= 0 && c->theta >= 0 && c->delta_p >= 0 && c->delta_v >= 0;
}

bool point_inside(const rich_config *c, double x, double y)
{
    if (c->boundary == RICH_BC_PERIODIC) return x >= c->x0 && x < c->x1 && y >= c->y0 && y < c->y1;
    return x > c->x0 && x < c->x1 && y > c->y0 && y < c->y1;
}

}  // namespace rich
using rich::point_inside;
using rich::valid_config;

struct rich_sim {
    rich_config cfg{};
    int32_t n = 0;
    std::vector<int32_t> perm;  // internal -> caller index
    // host copy of the points (internal order) for the host builder,
    // page-locked: x at [0, n), y at [n, 2n), then the dt of the sweep that
    // moved them
    rich::HBuf hpts;
    double *hx() const { return hpts.as<double>(); }
    double *hy() const { return hpts.as<double>() + n; }
    rich::MeshWork mw;  // (edge list built on the device: see tessellate)
    rich::HostMesh hm;  // the last mesh the host built
    // The mesh on the device (mesh[mcur]; an update writes the other while the
    // rest of the sweep reads this one): its sizes, and whether an update may
    // start from it
    rich::MeshStore mesh[2];
    int mcur = 0;
    rich::MeshSizes msz;
    bool mesh_on_device = false;
    rich::MeshUpdater updater;
    int64_t updates = 0;   // meshes made by it
    int missed = 0;        // updates in a row that left the mesh to the host
    int host_sweeps = 0;   // sweeps whose next mesh the host builds before another is tried
    rich::HBuf back;       // the step's dt and status, and the list builder's flag
    DBuf mesh_inst;        // the box and mesh_params
    rich::MeshStream mesh_stream;
    std::unique_ptr<rich::ThreadPool> pool;  // host threads of the tile-parallel tessellation
    rich_sim() { mw.host_edges = false; }
    double t = 0.0;
    int cur = 0;
    // time-centred scheme: 1 between its two sweeps (buffers [2] then hold
    // the half-step points and state)
    int tc_phase = 0;
    bool tess_current = false;
    bool pending = false;
    bool geometry_current = false;
    int diag_pts = 0;  // points buffer of the last completed sweep
    cudaStream_t stream = nullptr;
    cudaStream_t own_stream = nullptr;
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    bool profiling = false;
    cudaEvent_t kev[rich::NUM_STAGES + 1] = {};
    double kms[rich::NUM_STAGES] = {};
    double last_dt = 0.0;
    // device buffers
    DBuf x[3], y[3], U[3];
    DBuf A, o, W, cs, g, gl, alpha, w, tess, initW, rounding, p64, psrc;
    bool diagnostics = true;
    DBuf cell_of, unperm;  // internal cell of each caller index; reordered state for reads
    rich::HBuf read_host;  // (small reads)
    DBuf ccx, ccy, eL, emlx, emly, emrx, emry, enx, eny, eqx, eqy, F, ePM;
    DBuf scal;   // dtmin bits, dt, status
    DBuf instp;  // one InstParams
    rich::InstParams inst_host{};  // staging for the parameter upload

    ~rich_sim()
    {
        if (ev0) cudaEventDestroy(ev0);
        if (ev1) cudaEventDestroy(ev1);
        for (cudaEvent_t e : kev)
            if (e) cudaEventDestroy(e);
        if (own_stream) cudaStreamDestroy(own_stream);
    }

    template <class R> rich::SweepParams<R> params() const
    {
        rich::SweepParams<R> p{};
        p.inst = instp.as<rich::InstParams>();
        p.cell_inst = nullptr;
        p.n_inst = 1;
        p.diagnostics = diagnostics ? 1 : 0;
        p.motion = 1;
        p.n = n;
        mesh[mcur].describe(p, msz);
        // extrapolated fluxes: [cur] -> [1 - cur].  Time-centred: [cur] -> [2]
        // by half a step, then primitives and mesh of [2], update of [cur]
        // into [1 - cur]
        const int src = pts(), dst = next_pts();
        p.x = x[src].as<double>(); p.y = y[src].as<double>();
        p.xn = x[dst].as<double>(); p.yn = y[dst].as<double>();
        p.x0 = x[cur].as<double>(); p.y0 = y[cur].as<double>();
        p.ccx = ccx.as<double>(); p.ccy = ccy.as<double>(); p.A = A.as<double>();
        p.eL = eL.as<R>(); p.emlx = emlx.as<R>(); p.emly = emly.as<R>();
        p.emrx = emrx.as<R>(); p.emry = emry.as<R>();
        p.enx = enx.as<R>(); p.eny = eny.as<R>(); p.eqx = eqx.as<R>(); p.eqy = eqy.as<R>();
        p.ePM = ePM.as<rich::Vec4<R>>();
        p.U = U[src].as<double>(); p.Un = U[dst].as<double>(); p.U0 = U[cur].as<double>();
        p.W = W.as<rich::Vec4<R>>(); p.o = o.as<rich::Vec2<R>>(); p.cs = cs.as<R>();
        p.g = g.as<rich::Vec4<R>>(); p.gl = gl.as<rich::Vec4<R>>(); p.alpha = alpha.as<rich::Vec4<R>>();
        p.w = w.as<rich::Vec2<R>>();
        p.rounding = rounding.as<uint8_t>(); p.p64 = p64.as<double>();
        p.tess = tess.as<int32_t>(); p.F = F.as<rich::Vec4<R>>(); p.psrc = psrc.as<rich::Vec4<R>>();
        char *sc = scal.as<char>();
        p.dtmin_bits = reinterpret_cast<unsigned long long *>(sc);
        p.dt_out = reinterpret_cast<double *>(sc + 8);
        p.status = reinterpret_cast<int32_t *>(sc + 16);
        return p;
    }

    size_t rsize() const { return cfg.precision == RICH_FP32_SPLIT ? sizeof(float) : sizeof(double); }
    bool time_centred() const { return cfg.scheme == RICH_SCHEME_TIME_CENTRED; }
    // buffer of the points (and state) that the current mesh and sweep describe
    int pts() const { return tc_phase == 1 ? 2 : cur; }
    // buffer the sweep writes its moved points (and state) to
    int next_pts() const { return time_centred() && tc_phase == 0 ? 2 : 1 - cur; }

    // scheme parameters of this simulation with the time left to t_end
    rich::InstParams inst_params(double remaining, bool init = false) const
    {
        rich::InstParams ip{};
        ip.init = init ? 1 : 0;
        ip.gamma = cfg.gamma; ip.igm1 = 1.0 / (cfg.gamma - 1.0); ip.gamma_f = (float)ip.gamma; ip.igm1_f = (float)ip.igm1; ip.cfl = cfg.cfl; ip.chi = cfg.chi; ip.eta = cfg.eta; ip.theta = cfg.theta;
        ip.delta_v = cfg.delta_v; ip.delta_p = cfg.delta_p; ip.chi_f = (float)ip.chi; ip.theta_f = (float)ip.theta; ip.delta_v_f = (float)ip.delta_v;
        ip.x0 = cfg.x0; ip.x1 = cfg.x1; ip.y0 = cfg.y0; ip.y1 = cfg.y1;
        ip.remaining = remaining;
        ip.boundary = cfg.boundary; ip.motion = cfg.motion; ip.limiter = cfg.limiter;
        ip.phase = time_centred() ? 1 + tc_phase : 0;
        return ip;
    }

    // launch stage k of the sweep in the handle's precision (motion false:
    // the geometry stage leaves the mesh velocity and time step alone)
    void launch(int k, const double *init_W, double *Un_override = nullptr, bool motion = true) const
    {
        if (cfg.precision == RICH_FP32_SPLIT) {
            rich::SweepParams<float> p = params<float>();
            if (Un_override) p.Un = Un_override;
            p.motion = motion ? 1 : 0;
            rich::launch_stage<float>(k, p, init_W, stream);
        } else {
            rich::SweepParams<double> p = params<double>();
            if (Un_override) p.Un = Un_override;
            p.motion = motion ? 1 : 0;
            rich::launch_stage<double>(k, p, init_W, stream);
        }
    }

    // the mesh update's input: the mesh on the device and new positions
    rich::MeshArrays mesh_arrays(int q) const
    {
        rich::MeshArrays a{};
        a.n = n;
        a.n_inst = 1;
        a.inst = mesh_inst.as<rich::InstParams>();
        a.x = x[q].as<double>();
        a.y = y[q].as<double>();
        a.cell_ptr = mesh[mcur].cell_ptr.as<int32_t>();
        a.slot_nb = mesh[mcur].slot_nb.as<int32_t>();
        a.ghost_src = mesh[mcur].ghost_src.as<int32_t>();
        a.ghost_img = mesh[mcur].ghost_img.as<int32_t>();
        a.split = cfg.precision == RICH_FP32_SPLIT;
        return a;
    }
    int32_t periodic() const { return cfg.boundary == RICH_BC_PERIODIC ? 1 : 0; }
};

namespace {

int alloc_cells(rich_sim *s)
{
    const size_t n = (size_t)s->n, d = sizeof(double), r = s->rsize();
    for (int k = 0; k < (s->time_centred() ? 3 : 2); k++) {
        CUDA_TRY(s->x[k].ensure(n * d));
        CUDA_TRY(s->y[k].ensure(n * d));
        CUDA_TRY(s->U[k].ensure(4 * n * d));
    }
    CUDA_TRY(s->A.ensure(n * d)); CUDA_TRY(s->o.ensure(2 * n * r));
    CUDA_TRY(s->W.ensure(4 * n * r)); CUDA_TRY(s->cs.ensure(n * r));
    CUDA_TRY(s->g.ensure(8 * n * r)); CUDA_TRY(s->gl.ensure(8 * n * r)); CUDA_TRY(s->alpha.ensure(4 * n * r));
    CUDA_TRY(s->w.ensure(2 * n * r)); CUDA_TRY(s->tess.ensure(n * 4)); CUDA_TRY(s->psrc.ensure(4 * n * r));
    CUDA_TRY(s->rounding.ensure(n)); CUDA_TRY(s->p64.ensure(n * d));
    CUDA_TRY(s->scal.ensure(64));
    CUDA_TRY(cudaMemsetAsync(s->scal.p, 0, 64, s->stream));
    CUDA_TRY(s->instp.ensure(sizeof(rich::InstParams)));
    CUDA_TRY(s->back.ensure(64));
    CUDA_TRY(s->mesh_inst.ensure(sizeof(rich::InstParams)));
    rich::InstParams ip = s->inst_params(0.0);
    rich::mesh_params(rich::BoxConfig{s->cfg.boundary, s->cfg.x0, s->cfg.x1, s->cfg.y0, s->cfg.y1}, s->n, ip);
    CUDA_TRY(cudaMemcpyAsync(s->mesh_inst.p, &ip, sizeof(ip), cudaMemcpyHostToDevice, s->stream));
    CUDA_TRY(cudaStreamSynchronize(s->stream));
    return RICH_OK;
}

// a0 on the host: the mesh of the points in hx, hy (the device mesh is
// then out of date until upload_mesh)
int build_mesh(rich_sim *s, rich_step_info *info)
{
    rich::Range range("rich tessellate (a0)");
    const double t1 = now_ms();
    rich::BoxConfig box{s->cfg.boundary, s->cfg.x0, s->cfg.x1, s->cfg.y0, s->cfg.y1};
    const int rc = rich::build_host_mesh(box, s->n, s->hx(), s->hy(), s->mw, s->hm, s->pool.get());
    if (info) info->tess_ms += now_ms() - t1;
    return rc ? mesh_rc(rc) : RICH_OK;
}

// Room for the geometry of a mesh of these sizes (which every sweep computes
// afresh; nothing enqueued may still use the arrays).
int reserve_geometry(rich_sim *s, const rich::MeshSizes &z)
{
    const size_t d = sizeof(double), r = s->rsize(), T = (size_t)z.tris + 1, E = (size_t)z.edges + 1;
    CUDA_TRY(s->ccx.ensure(T * d)); CUDA_TRY(s->ccy.ensure(T * d));
    for (DBuf *b : {&s->eL, &s->emlx, &s->emly, &s->emrx, &s->emry, &s->enx, &s->eny, &s->eqx, &s->eqy})
        CUDA_TRY(b->ensure(E * r));
    CUDA_TRY(s->F.ensure(4 * E * d));
    CUDA_TRY(s->ePM.ensure(4 * E * r));
    return RICH_OK;
}

void report_sizes(const rich_sim *s, rich_step_info *info)
{
    if (!info) return;
    info->n_ghost = s->msz.ghosts;
    info->n_tri = s->msz.tris;
    info->n_edges = s->msz.edges;
    info->n_slots = s->msz.slots;
}

// Sizes that the device's update takes.
bool updatable(const rich_sim *s) { return s->n >= rich::kMeshUpdateMin && s->n <= rich::kMeshUpdateMax; }

// upload of the host mesh; the triangle and edge lists are built on the
// device from the rings (the host sends each cell's first owned triangle
// and edge, and the ghosts' images)
int upload_mesh(rich_sim *s, rich_step_info *info)
{
    const double t2 = now_ms();
    const rich::HostMesh &m = s->hm;
    s->mesh_on_device = false;
    s->updater.forget();
    s->msz = rich::MeshSizes{m.g, m.n_tris, m.n_edges, (int32_t)m.slot_nb.size()};
    rich::MeshStore &d = s->mesh[s->mcur];
    CUDA_TRY(d.reserve(s->n, s->msz));
    int rc = reserve_geometry(s, s->msz);
    if (rc != RICH_OK) return rc;
    // (the other store too where updates follow, as far as there is memory: the
    // first one then has room)
    if (updatable(s) && s->cfg.motion != RICH_MESH_EULERIAN && s->host_sweeps == 0)
        CUDA_TRY(rich::unless_no_room(s->mesh[1 - s->mcur].reserve(s->n, s->msz)));
    CUDA_TRY(upload(d.gx, m.gx, s->stream));
    CUDA_TRY(upload(d.gy, m.gy, s->stream));
    CUDA_TRY(upload(d.ghost_src, m.ghost_src, s->stream));
    CUDA_TRY(upload(d.ghost_img, m.ghost_img, s->stream));
    CUDA_TRY(upload(d.ghost_xf, m.ghost_xf, s->stream));
    CUDA_TRY(upload(d.ghost_shift, m.ghost_shift, s->stream));
    CUDA_TRY(upload(d.cell_ptr, m.cell_ptr, s->stream));
    CUDA_TRY(upload(d.cell_order, m.cell_order, s->stream));
    CUDA_TRY(upload(d.slot_nb, m.slot_nb, s->stream));
    CUDA_TRY(upload(d.tri_off, m.tri_off, s->stream));
    CUDA_TRY(upload(d.edge_off, m.edge_off, s->stream));
    rich::MeshLists l = d.lists(s->n, s->periodic());
    l.bad = reinterpret_cast<int32_t *>(s->scal.as<char>() + 24);
    CUDA_TRY(cudaMemsetAsync(l.bad, 0, sizeof(int32_t), s->stream));
    CUDA_TRY(rich::launch_lists(l, true, s->stream));
    CUDA_TRY(cudaMemcpyAsync(s->back.p, l.bad, sizeof(int32_t), cudaMemcpyDeviceToHost, s->stream));
    CUDA_TRY(cudaStreamSynchronize(s->stream));
    if (*s->back.as<int32_t>()) return fail(RICH_ETESS, "the rings of the mesh do not close");
    s->tess_current = s->mesh_on_device = true;
    if (info) info->copy_ms += now_ms() - t2;
    report_sizes(s, info);
    return RICH_OK;
}

// Whether the mesh of new points can be an update of the one on the device.
bool can_update(const rich_sim *s)
{
    return s->mesh_on_device && updatable(s);
}

// An update left the mesh to the host.
void missed_update(rich_sim *s)
{
    s->updater.forget();
    // (the same points would fail again)
    s->mesh_on_device = false;
    s->missed++;
    s->host_sweeps = rich::host_sweeps_after(s->missed);
}

// Enqueue the update of the mesh for the points in buffers q, on the mesh
// stream after what the handle's stream holds by now; join_update makes the
// handle's stream continue after it.  Without memory for it nothing is
// enqueued, and `started` is false: the mesh is the host's, and the room that
// updates hold is given back.
int start_update(rich_sim *s, int q, bool &started)
{
    rich::MeshStream &u = s->mesh_stream;
    CUDA_TRY(cudaEventRecord(u.moved, s->stream));
    CUDA_TRY(cudaStreamWaitEvent(u.stream, u.moved, 0));
    const cudaError_t e = s->updater.start(s->mesh_arrays(q), s->mesh[1 - s->mcur].output(s->periodic()), u.stream);
    started = e == cudaSuccess;
    CUDA_TRY(rich::unless_no_room(e));
    if (!started) {
        s->mesh[1 - s->mcur].release();
        s->missed = std::max(s->missed, 1);
        missed_update(s);
        return RICH_OK;
    }
    CUDA_TRY(cudaEventRecord(u.done, u.stream));
    return RICH_OK;
}

int join_update(rich_sim *s)
{
    CUDA_TRY(cudaStreamWaitEvent(s->stream, s->mesh_stream.done, 0));
    return RICH_OK;
}

// After the handle's stream was waited for: the updated mesh made the current
// one (keep), or dropped.  Where it could not be made the host has to build
// the points' own.
int finish_update(rich_sim *s, int q, bool keep, rich_step_info *info)
{
    if (!keep) {
        s->updater.forget();
        return RICH_OK;
    }
    const rich::MeshArrays a = s->mesh_arrays(q);
    rich::MeshStore &to = s->mesh[1 - s->mcur];
    cudaStream_t st = s->mesh_stream.stream;
    rich::MeshResult r;
    CUDA_TRY(s->updater.settle(a, to.output(s->periodic()), r, st));
    if (r.state == rich::MeshResult::kGrow) {
        const cudaError_t e = to.reserve(s->n, r.sizes);
        CUDA_TRY(rich::unless_no_room(e));
        if (e == cudaSuccess) CUDA_TRY(s->updater.again(a, to.output(s->periodic()), r, st));
    }
    if (r.state != rich::MeshResult::kDone || r.flagged) {
        missed_update(s);
        return RICH_OK;
    }
    s->missed = 0;
    s->mcur = 1 - s->mcur;
    s->msz = r.sizes;
    s->updates++;
    s->tess_current = true;
    report_sizes(s, info);
    // (the next update's buffers have as much room as these)
    CUDA_TRY(rich::unless_no_room(s->mesh[1 - s->mcur].reserve(s->n, r.sizes)));
    return reserve_geometry(s, r.sizes);
}

// a0 for the current points: the mesh on the device updated, or else built on
// the host and its connectivity uploaded.  fetch_points false: the host copy
// of the points is current, and there is no mesh to update.
int tessellate(rich_sim *s, rich_step_info *info, bool fetch_points)
{
    if (fetch_points && can_update(s)) {
        const double t0 = now_ms();
        const int q = s->pts();
        bool started = false;
        int rc = start_update(s, q, started);
        if (rc == RICH_OK && started) rc = join_update(s);
        if (rc != RICH_OK) return rc;
        s->tess_current = false;
        CUDA_TRY(cudaStreamSynchronize(s->stream));
        if (started && (rc = finish_update(s, q, true, info)) != RICH_OK) return rc;
        if (info) info->tess_ms += now_ms() - t0;
        if (s->tess_current) return RICH_OK;
    }
    if (fetch_points) {
        const double t0 = now_ms();
        const int q = s->pts();
        CUDA_TRY(cudaMemcpyAsync(s->hx(), s->x[q].p, sizeof(double) * s->n, cudaMemcpyDeviceToHost, s->stream));
        CUDA_TRY(cudaMemcpyAsync(s->hy(), s->y[q].p, sizeof(double) * s->n, cudaMemcpyDeviceToHost, s->stream));
        CUDA_TRY(cudaStreamSynchronize(s->stream));
        if (info) info->copy_ms += now_ms() - t0;
    }
    s->tess_current = false;
    int rc = build_mesh(s, info);
    if (rc) return rc;
    return upload_mesh(s, info);
}

}  // namespace

extern "C" {

void rich_default_config(rich_config *c)
{
    if (!c) return;
    std::memset(c, 0, sizeof(*c));
    c->gamma = 5.0 / 3.0;
    c->cfl = 0.3;
    c->boundary = RICH_BC_PERIODIC;
    c->x0 = 0.0; c->x1 = 1.0; c->y0 = 0.0; c->y1 = 1.0;
    c->motion = RICH_MESH_LAGRANGIAN;
    c->chi = 0.15; c->eta = 0.02;
    c->theta = 0.5; c->delta_v = 0.2; c->delta_p = 0.7;
    c->limiter = RICH_LIM_SWITCHED;
    c->scheme = RICH_SCHEME_EXTRAPOLATED;
    c->precision = RICH_FP64;
}

const char *rich_strerror(int code)
{
    switch (code) {
    case RICH_OK: return "ok";
    case RICH_EINVAL: return "invalid argument";
    case RICH_EDUPLICATE: return "coincident generating points";
    case RICH_ETESS: return "tessellation failed";
    case RICH_ETOOFEW: return "too few points for the ghost band";
    case RICH_ENEGATIVE: return "non-positive mass or thermal energy, or a point left the box";
    case RICH_ENAN: return "non-finite value";
    case RICH_ENOMEM: return "out of memory";
    case RICH_ECUDA: return "CUDA error";
    case RICH_ENODEV: return "no CUDA device";
    case RICH_ESTATE: return "call not valid in the current state";
    default: return "unknown error";
    }
}

const char *rich_last_error(void) { return rich::last_error(); }

int64_t rich_num_cells(const rich_sim *s) { return s ? s->n : -1; }

// Shared by rich_init_mesh (f = primitives rho, vx, vy, p) and
// rich_init_conserved (f = extensive m, px, py, E at time t0, cells in the
// internal order `order` when given).
static int create_sim(const rich_config *cfg, int64_t n, const double *x, const double *y, const double *const f[4],
                      bool conserved, double t0, const int64_t *order, rich_sim **out)
{
    if (!out) return fail(RICH_EINVAL, "out is NULL");
    *out = nullptr;
    if (!valid_config(cfg)) return fail(RICH_EINVAL, "invalid configuration");
    if (n < 3 || n > (int64_t)1 << 30) return fail(RICH_EINVAL, "n must be in [3, 2^30]");
    if (!x || !y || !f[0] || !f[1] || !f[2] || !f[3]) return fail(RICH_EINVAL, "NULL input array");
    if (!std::isfinite(t0)) return fail(RICH_EINVAL, "bad start time");
    for (int64_t i = 0; i < n; i++) {
        if (!std::isfinite(x[i]) || !std::isfinite(y[i]) || !point_inside(cfg, x[i], y[i]))
            return fail(RICH_EINVAL, "point " + std::to_string(i) + " outside the box");
        bool good = std::isfinite(f[0][i]) && std::isfinite(f[1][i]) && std::isfinite(f[2][i]) && std::isfinite(f[3][i]);
        if (conserved) good = good && f[0][i] > 0 && 2.0 * f[0][i] * f[3][i] - (f[1][i] * f[1][i] + f[2][i] * f[2][i]) > 0;
        else good = good && f[0][i] > 0 && f[3][i] > 0;
        if (!good) return fail(RICH_EINVAL, "bad field values at point " + std::to_string(i));
    }
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) return fail(RICH_ENODEV, "no CUDA device");
    rich_sim *s = new (std::nothrow) rich_sim();
    if (!s) return fail(RICH_ENOMEM, "host allocation");
    s->cfg = *cfg;
    s->n = (int32_t)n;
    s->t = t0;
    s->pool.reset(new (std::nothrow) rich::ThreadPool((int)std::max(1u, std::thread::hardware_concurrency())));
    if (!s->pool) {
        delete s;
        return fail(RICH_ENOMEM, "host thread pool");
    }
    if (order) {
        // the caller's internal order (a checkpoint's): must be a permutation
        s->perm.resize(n);
        std::vector<char> seen(n, 0);
        for (int64_t k = 0; k < n; k++) {
            if (order[k] < 0 || order[k] >= n || seen[order[k]]) {
                delete s;
                return fail(RICH_EINVAL, "order is not a permutation");
            }
            seen[order[k]] = 1;
            s->perm[k] = (int32_t)order[k];
        }
    } else {
        // renumber cells along a Hilbert curve for locality
        rich::hilbert_order(s->n, x, y, s->perm);
    }
    int rc = RICH_OK;
    auto bail = [&](int code) { delete s; return code; };
    if (s->hpts.ensure((2 * (size_t)n + 1) * sizeof(double)) != cudaSuccess)
        return bail(fail(RICH_ENOMEM, "page-locked host points"));
    std::vector<double> Fh(4 * (size_t)n);
    double *hx = s->hx(), *hy = s->hy();
    for (int32_t k = 0; k < s->n; k++) {
        int32_t u = s->perm[k];
        hx[k] = x[u];
        hy[k] = y[u];
        for (int c = 0; c < 4; c++) Fh[(size_t)c * n + k] = f[c][u];
    }
    if (cudaStreamCreateWithFlags(&s->own_stream, cudaStreamNonBlocking) != cudaSuccess)
        return bail(fail(RICH_ECUDA, "stream creation failed"));
    s->stream = s->own_stream;
    if (cudaEventCreate(&s->ev0) != cudaSuccess || cudaEventCreate(&s->ev1) != cudaSuccess ||
        s->mesh_stream.create() != cudaSuccess)
        return bail(fail(RICH_ECUDA, "event creation failed"));
    if ((rc = alloc_cells(s)) != RICH_OK) return bail(rc);
    if (s->x[0].ensure(n * 8) != cudaSuccess) return bail(fail(RICH_ENOMEM, "device points"));
    std::vector<int32_t> cell_of(n);
    for (int32_t k = 0; k < s->n; k++) cell_of[s->perm[k]] = k;
    if (upload(s->cell_of, cell_of, s->stream) != cudaSuccess) return bail(fail(RICH_ENOMEM, "device order"));
    cudaMemcpyAsync(s->x[0].p, hx, n * 8, cudaMemcpyHostToDevice, s->stream);
    cudaMemcpyAsync(s->y[0].p, hy, n * 8, cudaMemcpyHostToDevice, s->stream);
    if ((rc = tessellate(s, nullptr, false)) != RICH_OK) return bail(rc);
    if (conserved) {
        if (cudaMemcpyAsync(s->U[0].p, Fh.data(), 4 * n * 8, cudaMemcpyHostToDevice, s->stream) != cudaSuccess)
            return bail(fail(RICH_ECUDA, "state upload"));
    } else {
        if (s->initW.ensure(4 * n * 8) != cudaSuccess) return bail(fail(RICH_ENOMEM, "device primitives"));
        cudaMemcpyAsync(s->initW.p, Fh.data(), 4 * n * 8, cudaMemcpyHostToDevice, s->stream);
        s->inst_host = s->inst_params(0.0, true);
        if (cudaMemcpyAsync(s->instp.p, &s->inst_host, sizeof(rich::InstParams), cudaMemcpyHostToDevice,
                            s->stream) != cudaSuccess)
            return bail(fail(RICH_ECUDA, "parameter upload"));
        for (int k = 0; k < rich::GEOMETRY_STAGES; k++) s->launch(k, s->initW.as<double>(), s->U[0].as<double>());
    }
    cudaError_t e = cudaStreamSynchronize(s->stream);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return bail(fail(RICH_ECUDA, std::string("init: ") + cudaGetErrorString(e)));
    s->geometry_current = false;  // W not yet derived from U
    *out = s;
    return RICH_OK;
}

int rich_init_mesh(const rich_config *cfg, int64_t n, const double *x, const double *y, const double *rho,
                   const double *vx, const double *vy, const double *p, rich_sim **out)
{
    const double *f[4] = {rho, vx, vy, p};
    return create_sim(cfg, n, x, y, f, false, 0.0, nullptr, out);
}

int rich_init_conserved(const rich_config *cfg, int64_t n, const double *x, const double *y, const double *m,
                        const double *px, const double *py, const double *E, double t, const int64_t *order,
                        rich_sim **out)
{
    const double *f[4] = {m, px, py, E};
    return create_sim(cfg, n, x, y, f, true, t, order, out);
}

int rich_get_order(const rich_sim *s, int64_t n, int64_t *order)
{
    if (!s || n != s->n || !order) return fail(RICH_EINVAL, "bad arguments");
    for (int32_t k = 0; k < s->n; k++) order[k] = s->perm[k];
    return RICH_OK;
}

double rich_time(const rich_sim *s) { return s ? s->t : -1.0; }

void rich_destroy(rich_sim *s)
{
    if (!s) return;
    if (s->stream) cudaStreamSynchronize(s->stream);
    delete s;
}

int rich_set_stream(rich_sim *s, void *stream)
{
    if (!s) return fail(RICH_EINVAL, "NULL handle");
    CUDA_TRY(cudaStreamSynchronize(s->stream));
    s->stream = stream ? static_cast<cudaStream_t>(stream) : s->own_stream;
    return RICH_OK;
}

int rich_set_diagnostics(rich_sim *s, int32_t on)
{
    if (!s) return fail(RICH_EINVAL, "NULL handle");
    if (s->pending) return fail(RICH_ESTATE, "a sweep is pending; call rich_sync first");
    s->diagnostics = on != 0;
    return RICH_OK;
}

int rich_set_profiling(rich_sim *s, int32_t on)
{
    if (!s) return fail(RICH_EINVAL, "NULL handle");
    if (on && !s->kev[0])
        for (cudaEvent_t &e : s->kev) CUDA_TRY(cudaEventCreate(&e));
    s->profiling = on != 0;
    return RICH_OK;
}

int rich_kernel_times(rich_sim *s, int32_t cap, double *ms, int32_t *count)
{
    if (!s || !count) return fail(RICH_EINVAL, "bad arguments");
    *count = rich::NUM_STAGES;
    if (!s->profiling) return fail(RICH_ESTATE, "profiling is off");
    for (int k = 0; k < rich::NUM_STAGES && k < cap; k++) ms[k] = s->kms[k];
    return RICH_OK;
}

const char *rich_kernel_name(int32_t k) { return rich::stage_name(k); }

int rich_tessellate(rich_sim *s, rich_step_info *info)
{
    if (!s) return fail(RICH_EINVAL, "NULL handle");
    if (s->pending) return fail(RICH_ESTATE, "a sweep is pending; call rich_sync first");
    return tessellate(s, info, true);
}

// What a sweep starts once the points are moved: nothing, the update of the
// mesh for them, or their copy (and the dt's) to the host, which builds it.
enum class NextMesh { none, update, host };

// The moved points in buffers q and the dt to the host, on the mesh stream.
static int start_read(rich_sim *s, int q)
{
    rich::MeshStream &u = s->mesh_stream;
    const size_t bytes = (size_t)s->n * sizeof(double);
    CUDA_TRY(cudaEventRecord(u.moved, s->stream));
    CUDA_TRY(cudaStreamWaitEvent(u.stream, u.moved, 0));
    CUDA_TRY(cudaMemcpyAsync(s->hx(), s->x[q].p, bytes, cudaMemcpyDeviceToHost, u.stream));
    CUDA_TRY(cudaMemcpyAsync(s->hy(), s->y[q].p, bytes, cudaMemcpyDeviceToHost, u.stream));
    CUDA_TRY(cudaMemcpyAsync(s->hy() + s->n, s->scal.as<char>() + 8, 8, cudaMemcpyDeviceToHost, u.stream));
    CUDA_TRY(cudaEventRecord(u.done, u.stream));
    return RICH_OK;
}

// (next: what was started)
static int launch_sweep(rich_sim *s, double t_end, NextMesh &next)
{
    rich::Range range("rich sweep launch (a1-a9)");
    if (!s) return fail(RICH_EINVAL, "NULL handle");
    if (!s->tess_current) return fail(RICH_ESTATE, "no current tessellation");
    if (s->pending) return fail(RICH_ESTATE, "a sweep is pending; call rich_sync first");
    if (!(t_end > s->t)) return fail(RICH_EINVAL, "t_end must exceed the current time");
    s->inst_host = s->inst_params(t_end - s->t);
    CUDA_TRY(cudaMemcpyAsync(s->instp.p, &s->inst_host, sizeof(rich::InstParams), cudaMemcpyHostToDevice, s->stream));
    CUDA_TRY(cudaEventRecord(s->ev0, s->stream));
    for (int k = 0; k < rich::NUM_STAGES; k++) {
        if (s->profiling) CUDA_TRY(cudaEventRecord(s->kev[k], s->stream));
        s->launch(k, nullptr);
        if (k != rich::K_ADVANCE) continue;
        int rc = RICH_OK;
        if (next == NextMesh::update) {
            bool started = false;
            rc = start_update(s, s->next_pts(), started);
            if (!started) next = NextMesh::host;
        }
        if (rc == RICH_OK && next == NextMesh::host) rc = start_read(s, s->next_pts());
        if (rc != RICH_OK) return rc;
    }
    if (s->profiling) CUDA_TRY(cudaEventRecord(s->kev[rich::NUM_STAGES], s->stream));
    CUDA_TRY(cudaGetLastError());
    CUDA_TRY(cudaEventRecord(s->ev1, s->stream));
    s->pending = true;
    return RICH_OK;
}

int rich_sweep(rich_sim *s, double t_end)
{
    NextMesh next = NextMesh::none;
    return launch_sweep(s, t_end, next);
}

// The sweep's dt and status, into page-locked memory (dt, then the status)
static int fetch_result(rich_sim *s)
{
    CUDA_TRY(cudaMemcpyAsync(s->back.as<double>() + 1, s->scal.as<char>() + 8, 12, cudaMemcpyDeviceToHost, s->stream));
    return RICH_OK;
}

// rich_sync after fetch_result
static int wait_sweep(rich_sim *s, rich_step_info *info)
{
    double t0 = now_ms();
    char *sc = s->scal.as<char>();
    const double *dt_host = s->back.as<double>() + 1;
    const int32_t *status_host = reinterpret_cast<const int32_t *>(dt_host + 1);
    CUDA_TRY(cudaStreamSynchronize(s->stream));
    const double dt = *dt_host;
    const int32_t status = *status_host;
    s->pending = false;
    float ms = 0.0f;
    cudaEventElapsedTime(&ms, s->ev0, s->ev1);
    if (s->profiling)
        for (int k = 0; k < rich::NUM_STAGES; k++) {
            float km = 0.0f;
            cudaEventElapsedTime(&km, s->kev[k], s->kev[k + 1]);
            s->kms[k] = km;
        }
    if (info) {
        info->sweep_ms += ms;
        info->copy_ms += now_ms() - t0;
    }
    s->geometry_current = true;  // diagnostics describe this sweep
    s->diag_pts = s->pts();
    if (status) {
        CUDA_TRY(cudaMemsetAsync(sc + 16, 0, 4, s->stream));
        CUDA_TRY(cudaStreamSynchronize(s->stream));
        if (s->tc_phase == 1) {
            // the full step failed: start the step again from [cur]
            s->tc_phase = 0;
            s->tess_current = false;
        }
        if (status & rich::ST_NAN) return fail(RICH_ENAN, "non-finite state after the step");
        if (status & rich::ST_LEFT_BOX) return fail(RICH_ENEGATIVE, "a generating point left the box");
        return fail(RICH_ENEGATIVE, "non-positive mass or thermal energy after the step");
    }
    s->last_dt = dt;
    s->tess_current = false;
    if (s->time_centred() && s->tc_phase == 0) {
        // half step done: the next sweep is the full step on the half-step mesh
        s->tc_phase = 1;
        return RICH_OK;
    }
    s->tc_phase = 0;
    s->cur = 1 - s->cur;
    s->t += dt;
    if (info) {
        info->steps_done += 1;
        info->t = s->t;
        info->dt_last = dt;
    }
    return RICH_OK;
}

int rich_sync(rich_sim *s, rich_step_info *info)
{
    rich::Range range("rich sync");
    if (!s) return fail(RICH_EINVAL, "NULL handle");
    if (!s->pending) return fail(RICH_ESTATE, "no sweep pending");
    const int rc = fetch_result(s);
    return rc != RICH_OK ? rc : wait_sweep(s, info);
}

// One sweep of rich_step: the update of the mesh for the moved points runs on
// the mesh stream beside the gradients, fluxes and update, from when the
// points are there (those stages leave the memory pipes and the FP32 and
// integer units idle, which the update lives on), and one wait serves both.
// A failed sweep drops the updated mesh; one that the update cannot make is
// left to the next tessellation.  Where updates keep failing, and for sizes
// that they do not take, the host builds the mesh beside those stages instead,
// unless the sweep ends the run at t_end.
static int step_sweep(rich_sim *s, double t_end, rich_step_info *info)
{
    const int q = s->next_pts();
    // (a static mesh's points stay where they are, bit for bit: x + dt 0)
    const bool still = s->cfg.motion == RICH_MESH_EULERIAN;
    NextMesh next = still                                  ? NextMesh::none
                    : can_update(s) && s->host_sweeps == 0 ? NextMesh::update
                                                            : NextMesh::host;
    if (next == NextMesh::host && s->host_sweeps > 0) s->host_sweeps--;
    int rc = launch_sweep(s, t_end, next);
    if (rc != RICH_OK) return rc;
    // (the sweep's result is copied while the update still runs)
    if ((rc = fetch_result(s)) != RICH_OK) return rc;
    if (next == NextMesh::update && (rc = join_update(s)) != RICH_OK) return rc;
    bool built = false;
    if (next == NextMesh::host) {
        const double t0 = now_ms();
        CUDA_TRY(cudaEventSynchronize(s->mesh_stream.done));
        if (info) info->copy_ms += now_ms() - t0;
        // the half-step points always get a mesh; after a full step, the
        // points get one unless the step lands on t_end
        if ((s->time_centred() && s->tc_phase == 0) || s->hy()[s->n] < t_end - s->t) {
            s->tess_current = false;
            // (a mesh that cannot be built is reported by the next
            // tessellation of the same points)
            built = build_mesh(s, info) == RICH_OK;
        }
    }
    rc = wait_sweep(s, info);
    if (still && rc == RICH_OK) {
        s->tess_current = true;
        report_sizes(s, info);
    }
    if (next == NextMesh::host) {
        // (after a failed sweep the host's mesh is not that of the points)
        if (rc != RICH_OK || !built) return rc;
        return upload_mesh(s, info);
    }
    if (next != NextMesh::update) return rc;
    const double t0 = now_ms();
    const int urc = finish_update(s, q, rc == RICH_OK, info);
    // (what the update takes beyond the end of the sweep)
    float ms = 0.0f;
    if (info && cudaEventElapsedTime(&ms, s->ev1, s->mesh_stream.done) == cudaSuccess && ms > 0.0f) info->tess_ms += ms;
    if (info) info->tess_ms += now_ms() - t0;
    return rc != RICH_OK ? rc : urc;
}

int rich_step(rich_sim *s, int32_t max_steps, double t_end, rich_step_info *info)
{
    rich::Range range("rich step");
    if (!s) return fail(RICH_EINVAL, "NULL handle");
    if (s->pending) return fail(RICH_ESTATE, "a sweep is pending; call rich_sync first");
    if (info) std::memset(info, 0, sizeof(*info));
    for (int32_t k = 0; k < max_steps; k++) {
        if (!(s->t < t_end)) break;
        int rc;
        if (!s->tess_current && (rc = tessellate(s, info, true)) != RICH_OK) return rc;
        double before = s->t;
        if ((rc = step_sweep(s, t_end, info)) != RICH_OK) return rc;
        if (s->tc_phase == 1) {
            // time-centred: the full step on the mesh of the half-step points
            // (meshed again here, to report its error, if the early build failed)
            if (!s->tess_current && (rc = tessellate(s, info, true)) != RICH_OK) return rc;
            if ((rc = step_sweep(s, t_end, info)) != RICH_OK) return rc;
        }
        if (s->last_dt >= t_end - before) s->t = t_end;  // landed on t_end
        if (info) info->t = s->t;
    }
    if (info) {
        info->t = s->t;
        info->dt_last = s->last_dt;
    }
    return RICH_OK;
}

static int ensure_geometry(rich_sim *s)
{
    if (s->pending) return fail(RICH_ESTATE, "a sweep is pending; call rich_sync first");
    if (!s->tess_current) {
        int rc = tessellate(s, nullptr, true);
        if (rc) return rc;
    }
    for (int k = 0; k < rich::GEOMETRY_STAGES; k++) s->launch(k, nullptr, nullptr, false);
    CUDA_TRY(cudaGetLastError());
    // the cell geometry and primitives now describe the current points (once
    // the stream gets there)
    s->geometry_current = true;
    s->diag_pts = s->pts();
    return RICH_OK;
}

static void unpermute(const rich_sim *s, const double *internal, double *out)
{
    for (int32_t k = 0; k < s->n; k++) out[s->perm[k]] = internal[k];
}

static int fetch(rich_sim *s, const void *dev, std::vector<double> &h, size_t count)
{
    h.resize(count);
    CUDA_TRY(cudaMemcpyAsync(h.data(), dev, count * 8, cudaMemcpyDeviceToHost, s->stream));
    CUDA_TRY(cudaStreamSynchronize(s->stream));
    return RICH_OK;
}

// fetch count values stored in the handle's reconstruction precision
static int fetch_r(rich_sim *s, const void *dev, std::vector<double> &h, size_t count)
{
    if (s->rsize() == sizeof(double)) return fetch(s, dev, h, count);
    std::vector<float> f(count);
    CUDA_TRY(cudaMemcpyAsync(f.data(), dev, count * 4, cudaMemcpyDeviceToHost, s->stream));
    CUDA_TRY(cudaStreamSynchronize(s->stream));
    h.assign(f.begin(), f.end());
    return RICH_OK;
}

// Where a read of `fields` fields is gathered: page-locked memory for small
// ones (each copy to pageable memory costs about 8 us whatever its size), else
// the device (the host then copies nothing itself).  Reads of the conserved state
// take 24 and 63 us for 4,096 cells, 60 and 68 for 16,384, 69 and 68 for 19,600
// (0.90 MB), 110 and 72 for 32,761; of the state (seven fields) 83 and 88 us for
// 16,384, 96 and 92 for 19,600 (1.05 MB).  (Null without memory for it: the host
// reorders then.)
static int read_buffer(rich_sim *s, int fields, double **buf, bool *host)
{
    const size_t bytes = (size_t)s->n * fields * 8;
    *host = bytes <= ((size_t)7 << 17);
    CUDA_TRY(rich::unless_no_room(*host ? s->read_host.ensure(bytes) : s->unperm.ensure(bytes)));
    *buf = *host ? s->read_host.as<double>() : s->unperm.as<double>();
    return RICH_OK;
}

// Fields (null ones skipped) through host memory, field by field.
static int read_fields(rich_sim *s, const double *const *src, double *const *outs, int fields)
{
    std::vector<double> h;
    for (int f = 0; f < fields; f++) {
        if (!outs[f]) continue;
        const int rc = fetch(s, src[f], h, (size_t)s->n);
        if (rc) return rc;
        unpermute(s, h.data(), outs[f]);
    }
    return RICH_OK;
}

// From there to the caller's arrays (null ones skipped).  Waits.
static int copy_out(rich_sim *s, const double *buf, bool host, double *const *outs, int fields)
{
    const size_t N = (size_t)s->n;
    for (int f = 0; f < fields && !host; f++)
        if (outs[f]) CUDA_TRY(cudaMemcpyAsync(outs[f], buf + f * N, N * 8, cudaMemcpyDeviceToHost, s->stream));
    CUDA_TRY(cudaStreamSynchronize(s->stream));
    for (int f = 0; f < fields && host; f++)
        if (outs[f]) std::memcpy(outs[f], buf + f * N, N * 8);
    return RICH_OK;
}

int rich_get_state(rich_sim *s, int64_t n, double *x, double *y, double *rho, double *vx, double *vy, double *p,
                   double *area)
{
    if (!s || n != s->n) return fail(RICH_EINVAL, "bad handle or size");
    int rc = ensure_geometry(s);
    if (rc) return rc;
    // put in the caller's order on the device, then copied straight into the
    // caller's arrays with one wait (on the host the reordering took 2.4 ms of
    // a 3.0 ms step and read at 262,144 cells)
    const int q = s->pts();
    double *outs[7] = {x, y, rho, vx, vy, p, area};
    double *st;
    bool host;
    if ((rc = read_buffer(s, 7, &st, &host))) return rc;
    if (!st) {
        const double *src[3] = {s->x[q].as<double>(), s->y[q].as<double>(), s->A.as<double>()};
        double *const to[3] = {x, y, area};
        if ((rc = read_fields(s, src, to, 3))) return rc;
        std::vector<double> h, W;
        if ((rc = fetch_r(s, s->W.p, W, 4 * (size_t)n))) return rc;
        h.resize((size_t)n);
        for (int c = 0; c < 4; c++) {
            if (!outs[2 + c]) continue;
            for (size_t k = 0; k < (size_t)n; k++) h[k] = W[4 * k + c];
            unpermute(s, h.data(), outs[2 + c]);
        }
        return RICH_OK;
    }
    CUDA_TRY(rich::launch_unpermute_state(s->n, s->cell_of.as<int32_t>(), s->x[q].as<double>(), s->y[q].as<double>(),
                                          s->W.p, s->rsize() == sizeof(float), s->A.as<double>(), st, s->stream));
    return copy_out(s, st, host, outs, 7);
}

int rich_get_conserved(rich_sim *s, int64_t n, double *x, double *y, double *m, double *px, double *py, double *E)
{
    if (!s || n != s->n) return fail(RICH_EINVAL, "bad handle or size");
    if (s->pending) return fail(RICH_ESTATE, "a sweep is pending; call rich_sync first");
    const size_t N = (size_t)s->n;
    const int q = s->pts();
    // points and state put in the caller's order on the device, then copied
    // straight into the caller's arrays with one wait
    double *outs[6] = {x, y, m, px, py, E};
    const double *src[6] = {s->x[q].as<double>(), s->y[q].as<double>(), s->U[q].as<double>(),
                            s->U[q].as<double>() + N, s->U[q].as<double>() + 2 * N, s->U[q].as<double>() + 3 * N};
    for (int f = 0; f < 6; f++)
        if (!outs[f]) src[f] = nullptr;
    double *st;
    bool host;
    int rc = read_buffer(s, 6, &st, &host);
    if (rc) return rc;
    if (!st) return read_fields(s, src, outs, 6);
    CUDA_TRY(rich::launch_unpermute(s->n, s->cell_of.as<int32_t>(), src, st, s->stream));
    return copy_out(s, st, host, outs, 6);
}

int rich_get_field(rich_sim *s, int32_t f, int64_t n, double *out)
{
    if (!s || n != s->n || !out) return fail(RICH_EINVAL, "bad arguments");
    if (s->pending) return fail(RICH_ESTATE, "a sweep is pending; call rich_sync first");
    const size_t N = (size_t)s->n;
    std::vector<double> h, h2;
    int rc;
    // the diagnostics refer to the points of the last sweep (or of the last
    // geometry pass on the current points)
    const int prev = s->geometry_current ? s->diag_pts : s->pts();
    // gather component c of an array-of-structures field with `stride` values per cell
    auto comp_of = [&](const DBuf &b, int stride, int c) {
        int r2 = fetch_r(s, b.p, h2, stride * N);
        if (r2) return r2;
        h.resize(N);
        for (size_t k = 0; k < N; k++) h[k] = h2[stride * k + c];
        return RICH_OK;
    };
    if (f == 0) rc = fetch(s, s->A.p, h, N);
    else if (f == 1 || f == 2) {
        if ((rc = comp_of(s->o, 2, f - 1))) return rc;
        std::vector<double> xs;
        rc = fetch(s, (f == 1 ? s->x[prev] : s->y[prev]).p, xs, N);
        for (size_t k = 0; k < N; k++) h[k] += xs[k];
    } else if (f >= 3 && f <= 6) rc = comp_of(s->W, 4, f - 3);
    else if (f == 7) rc = fetch_r(s, s->cs.p, h, N);
    else if (f >= 8 && f <= 23) rc = comp_of(f < 16 ? s->g : s->gl, 8, (f - 8) % 8);
    else if (f == 24 || f == 25) rc = comp_of(s->w, 2, f - 24);
    else if (f == 26) {
        std::vector<int32_t> ti(N);
        CUDA_TRY(cudaMemcpyAsync(ti.data(), s->tess.p, N * 4, cudaMemcpyDeviceToHost, s->stream));
        CUDA_TRY(cudaStreamSynchronize(s->stream));
        h.resize(N);
        for (size_t k = 0; k < N; k++) h[k] = ti[k];
        rc = RICH_OK;
    } else if (f >= 27 && f <= 30) rc = comp_of(s->alpha, 4, f - 27);
    else if (f == 31) {
        h.assign(N, s->last_dt);
        rc = RICH_OK;
    } else
        return fail(RICH_EINVAL, "unknown field");
    if (rc) return rc;
    unpermute(s, h.data(), out);
    return RICH_OK;
}

int rich_delaunay_host(int64_t n, const double *x, const double *y, int64_t cap, int32_t *tris, int64_t *ntri)
{
    if (n < 1 || !x || !y || !ntri) return fail(RICH_EINVAL, "bad arguments");
    rich::Delaunay dt;
    int rc = dt.build(x, y, (int32_t)n);
    if (rc == -2) return fail(RICH_EDUPLICATE, "two points coincide");
    if (rc) return fail(RICH_ETESS, "triangulation failed");
    *ntri = (int64_t)dt.tris.size();
    if (cap < *ntri || !tris) return fail(RICH_EINVAL, "capacity too small");
    for (size_t t = 0; t < dt.tris.size(); t++)
        for (int k = 0; k < 3; k++) tris[3 * t + k] = dt.tris[t].v[k];
    return RICH_OK;
}

int rich_rings_host(const rich_config *cfg, int64_t n, const double *x, const double *y, int64_t cap, int64_t *ptr,
                    double *nbx, double *nby, int64_t *nbsrc, int64_t *nslots)
{
    if (!valid_config(cfg) || n < 3 || !x || !y || !nslots || !ptr) return fail(RICH_EINVAL, "bad arguments");
    for (int64_t i = 0; i < n; i++)
        if (!point_inside(cfg, x[i], y[i])) return fail(RICH_EINVAL, "point outside the box");
    rich::MeshWork mw;
    rich::HostMesh m;
    rich::BoxConfig box{cfg->boundary, cfg->x0, cfg->x1, cfg->y0, cfg->y1};
    rich::ThreadPool pool((int)std::max(1u, std::thread::hardware_concurrency()));
    int rc = rich::build_host_mesh(box, (int32_t)n, x, y, mw, m, &pool);
    if (rc) return mesh_rc(rc);
    *nslots = (int64_t)m.slot_nb.size();
    for (int64_t i = 0; i <= n; i++) ptr[i] = m.cell_ptr[i];
    if (cap < *nslots || !nbx || !nby || !nbsrc) return fail(RICH_EINVAL, "capacity too small");
    for (size_t s = 0; s < m.slot_nb.size(); s++) {
        int32_t q = m.slot_nb[s];
        if (q < n) { nbx[s] = x[q]; nby[s] = y[q]; nbsrc[s] = q; }
        else { nbx[s] = m.gx[q - n]; nby[s] = m.gy[q - n]; nbsrc[s] = m.ghost_src[q - n]; }
    }
    return RICH_OK;
}

int rich_tess_phases(const rich_sim *s, double *ms)
{
    if (!s || !ms) return fail(RICH_EINVAL, "bad arguments");
    for (int k = 0; k < 4; k++) ms[k] = s->mw.phase_ms[k];
    return RICH_OK;
}

int rich_edge_list_check(const rich_config *cfg, int64_t n, const double *x, const double *y, int64_t *edges,
                         int64_t *mismatched)
{
    if (!valid_config(cfg) || n < 3 || n > INT32_MAX || !x || !y || !edges || !mismatched)
        return fail(RICH_EINVAL, "bad arguments");
    for (int64_t i = 0; i < n; i++)
        if (!point_inside(cfg, x[i], y[i])) return fail(RICH_EINVAL, "point outside the box");
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) return fail(RICH_ENODEV, "no CUDA device");
    const rich::BoxConfig box{cfg->boundary, cfg->x0, cfg->x1, cfg->y0, cfg->y1};
    rich::ThreadPool pool((int)std::max(1u, std::thread::hardware_concurrency()));
    rich::MeshWork mw;  // host_edges: the host builds the reference lists too
    rich::HostMesh m;
    int rc = rich::build_host_mesh(box, (int32_t)n, x, y, mw, m, &pool);
    if (rc) return mesh_rc(rc);
    // the same points as a simulation builds them: rings and tri_off only
    rich::MeshWork mw2;
    mw2.host_edges = false;
    rich::HostMesh m2;
    rc = rich::build_host_mesh(box, (int32_t)n, x, y, mw2, m2, &pool);
    if (rc) return mesh_rc(rc);
    if (m2.slot_nb != m.slot_nb || m2.cell_ptr != m.cell_ptr) return fail(RICH_ETESS, "rings differ between builds");
    const size_t S = m.slot_nb.size(), E = (size_t)m.n_edges, T2 = (size_t)m2.n_tris;
    cudaStream_t st = nullptr;
    CUDA_TRY(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking));
    DBuf cell_ptr, slot_nb, gsrc, gshift, eoff, slot_edge, el, er, eta, etb, bad, toff, dtri, dslot_tri;
    auto up = [&](DBuf &d, const std::vector<int32_t> &h) -> cudaError_t {
        cudaError_t e = d.ensure((h.size() + 1) * sizeof(int32_t));
        if (e == cudaSuccess && !h.empty())
            e = cudaMemcpyAsync(d.p, h.data(), h.size() * sizeof(int32_t), cudaMemcpyHostToDevice, st);
        return e;
    };
    std::vector<int32_t> dse(S), del(E), der(E), deta(E), detb(E), dt(3 * T2), dst(S);
    int32_t bad_h = 0;
    cudaError_t e = up(cell_ptr, m.cell_ptr);
    if (e == cudaSuccess) e = up(slot_nb, m.slot_nb);
    if (e == cudaSuccess) e = up(gsrc, m.ghost_src);
    if (e == cudaSuccess) e = up(gshift, m.ghost_shift);
    if (e == cudaSuccess) e = up(eoff, m.edge_off);
    if (e == cudaSuccess) e = up(toff, m2.tri_off);
    // (every slot has to be written: an entry the builder leaves shows)
    for (DBuf *b : {&slot_edge, &dslot_tri}) {
        if (e == cudaSuccess) e = b->ensure((S + 1) * sizeof(int32_t));
        if (e == cudaSuccess) e = cudaMemsetAsync(b->p, 0xff, b->cap, st);
    }
    for (DBuf *b : {&el, &er, &eta, &etb}) if (e == cudaSuccess) e = b->ensure((E + 1) * sizeof(int32_t));
    if (e == cudaSuccess) e = bad.ensure(sizeof(int32_t));
    if (e == cudaSuccess) e = cudaMemsetAsync(bad.p, 0, sizeof(int32_t), st);
    if (e == cudaSuccess) e = dtri.ensure((3 * T2 + 3) * sizeof(int32_t));
    if (e == cudaSuccess) {
        rich::MeshLists l{};
        l.n = (int32_t)n;
        l.periodic = cfg->boundary == RICH_BC_PERIODIC ? 1 : 0;
        l.cell_ptr = cell_ptr.as<int32_t>(); l.slot_nb = slot_nb.as<int32_t>();
        l.tri_off = toff.as<int32_t>(); l.edge_off = eoff.as<int32_t>();
        l.ghost_src = gsrc.as<int32_t>(); l.ghost_shift = gshift.as<int32_t>();
        l.tri = dtri.as<int32_t>(); l.slot_tri = dslot_tri.as<int32_t>(); l.slot_edge = slot_edge.as<int32_t>();
        l.edge_l = el.as<int32_t>(); l.edge_r = er.as<int32_t>();
        l.edge_ta = eta.as<int32_t>(); l.edge_tb = etb.as<int32_t>();
        l.bad = bad.as<int32_t>();
        e = rich::launch_lists(l, true, st);
    }
    auto down = [&](std::vector<int32_t> &h, DBuf &d) {
        if (e == cudaSuccess && !h.empty())
            e = cudaMemcpyAsync(h.data(), d.p, h.size() * sizeof(int32_t), cudaMemcpyDeviceToHost, st);
    };
    down(dse, slot_edge);
    down(del, el);
    down(der, er);
    down(deta, eta);
    down(detb, etb);
    down(dt, dtri);
    down(dst, dslot_tri);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&bad_h, bad.p, sizeof(int32_t), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaStreamDestroy(st);
    if (e != cudaSuccess) return fail(RICH_ECUDA, cudaGetErrorString(e));
    int64_t bad_count = bad_h ? 1 : 0;
    for (size_t k = 0; k < S; k++) bad_count += dse[k] != m.slot_edge[k];
    // the device's triangle of every slot: the host's, vertex for vertex
    // (the numbering differs: the host's is per tile)
    for (size_t k = 0; k < S; k++) {
        const int32_t a = dst[k], h = m.slot_tri[k];
        if (a < 0 || (size_t)a >= T2) {
            bad_count++;
            continue;
        }
        for (int c = 0; c < 3; c++) bad_count += dt[3 * (size_t)a + c] != m.tri[3 * (size_t)h + c];
    }
    // (the edges' Voronoi vertices: the device's triangles, vertex for vertex)
    auto same_tri = [&](int32_t a, int32_t h) {
        if (a < 0 || (size_t)a >= T2) return false;
        for (int c = 0; c < 3; c++)
            if (dt[3 * (size_t)a + c] != m.tri[3 * (size_t)h + c]) return false;
        return true;
    };
    for (size_t k = 0; k < E; k++)
        bad_count += (del[k] != m.edge_l[k]) + (der[k] != m.edge_r[k]) + !same_tri(deta[k], m.edge_ta[k]) +
                     !same_tri(detb[k], m.edge_tb[k]);
    *edges = (int64_t)E;
    *mismatched = bad_count;
    return RICH_OK;
}

int rich_mesh_update_check(const rich_config *cfg, int64_t n, int32_t steps, const double *xs, const double *ys,
                           int32_t threads, int32_t *mismatched, int64_t *updated, int64_t *rebuilt,
                           int64_t *reinserted)
{
    if (!valid_config(cfg) || n < 3 || n > INT32_MAX || steps < 1 || !xs || !ys || !mismatched || !updated ||
        !rebuilt || !reinserted || threads < 1)
        return fail(RICH_EINVAL, "bad arguments");
    for (int64_t i = 0; i < (int64_t)steps * n; i++)
        if (!point_inside(cfg, xs[i], ys[i])) return fail(RICH_EINVAL, "point outside the box");
    const rich::BoxConfig box{cfg->boundary, cfg->x0, cfg->x1, cfg->y0, cfg->y1};
    rich::ThreadPool pool(threads);
    rich::MeshWork kept;
    // the same sequence as a simulation builds it (no host lists: the rings
    // are read off incrementally and copied where unchanged)
    rich::MeshWork kept_dev;
    kept_dev.host_edges = false;
    *mismatched = 0;
    // a triangle's vertices (smallest id first in both builds)
    auto tri_of = [](const rich::HostMesh &m, int32_t t) {
        return std::array<int32_t, 3>{m.tri[3 * (size_t)t], m.tri[3 * (size_t)t + 1], m.tri[3 * (size_t)t + 2]};
    };
    for (int32_t k = 0; k < steps; k++) {
        const double *x = xs + (size_t)k * n, *y = ys + (size_t)k * n;
        rich::HostMesh a, b, c;
        rich::MeshWork fresh;
        int rc = rich::build_host_mesh(box, (int32_t)n, x, y, kept, a, &pool);
        if (rc) return mesh_rc(rc);
        rc = rich::build_host_mesh(box, (int32_t)n, x, y, fresh, b, &pool);
        if (rc) return mesh_rc(rc);
        rc = rich::build_host_mesh(box, (int32_t)n, x, y, kept_dev, c, &pool);
        if (rc) return mesh_rc(rc);
        if (!(c.g == b.g && c.gx == b.gx && c.gy == b.gy && c.ghost_src == b.ghost_src && c.cell_ptr == b.cell_ptr &&
              c.slot_nb == b.slot_nb && c.edge_off == b.edge_off && c.n_edges == b.n_edges &&
              c.cell_order == b.cell_order && (int64_t)c.tri_off.size() == n + 1 && c.tri_off[n] == c.n_tris))
            (*mismatched)++;
        bool same = a.g == b.g && a.gx == b.gx && a.gy == b.gy && a.ghost_src == b.ghost_src &&
                    a.cell_ptr == b.cell_ptr && a.slot_nb == b.slot_nb && a.slot_edge == b.slot_edge &&
                    a.edge_l == b.edge_l && a.edge_r == b.edge_r && a.cell_order == b.cell_order &&
                    a.edge_off == b.edge_off && a.n_edges == b.n_edges && (size_t)b.n_edges == b.edge_l.size();
        // the per-cell first edges (what the device builder numbers from)
        // agree with the host's list: cell i owns edges [edge_off[i], edge_off[i + 1])
        for (int64_t i = 0; same && i < n; i++)
            for (int32_t e = b.edge_off[i]; same && e < b.edge_off[i + 1]; e++) same = b.edge_l[e] == (int32_t)i;
        for (size_t s = 0; same && s < a.slot_tri.size(); s++) same = tri_of(a, a.slot_tri[s]) == tri_of(b, b.slot_tri[s]);
        for (size_t e = 0; same && e < a.edge_ta.size(); e++)
            same = tri_of(a, a.edge_ta[e]) == tri_of(b, b.edge_ta[e]) && tri_of(a, a.edge_tb[e]) == tri_of(b, b.edge_tb[e]);
        if (!same) (*mismatched)++;
    }
    *updated = kept.kinetic_tiles;
    *rebuilt = kept.fresh_tiles;
    *reinserted = kept.reinserted;
    return RICH_OK;
}

// entries of the device mesh update's output that differ from a fresh host build
static int64_t mesh_differences(const rich::HostMesh &a, const rich::HostMesh &b)
{
    int64_t bad = 0;
    auto cmp = [&](const auto &u, const auto &v) {
        if (u.size() != v.size()) {
            bad++;
            return;
        }
        for (size_t k = 0; k < u.size(); k++) bad += u[k] != v[k];
    };
    cmp(a.cell_ptr, b.cell_ptr);
    cmp(a.slot_nb, b.slot_nb);
    cmp(a.tri_off, b.tri_off);
    cmp(a.edge_off, b.edge_off);
    cmp(a.cell_order, b.cell_order);
    cmp(a.gx, b.gx);
    cmp(a.gy, b.gy);
    cmp(a.ghost_src, b.ghost_src);
    cmp(a.ghost_xf, b.ghost_xf);
    cmp(a.ghost_shift, b.ghost_shift);
    cmp(a.ghost_img, b.ghost_img);
    return bad;
}

int rich_device_update_check(const rich_config *cfg, int64_t n, int32_t steps, const double *xs, const double *ys,
                             int64_t *mismatched, int64_t *updated, int64_t *recomputed)
{
    if (!valid_config(cfg) || n < 3 || n > rich::kMeshUpdateMax || steps < 1 || !xs || !ys || !mismatched || !updated ||
        !recomputed)
        return fail(RICH_EINVAL, "bad arguments");
    for (int64_t i = 0; i < (int64_t)steps * n; i++)
        if (!point_inside(cfg, xs[i], ys[i])) return fail(RICH_EINVAL, "point outside the box");
    const rich::BoxConfig box{cfg->boundary, cfg->x0, cfg->x1, cfg->y0, cfg->y1};
    rich::ThreadPool pool((int)std::max(1u, std::thread::hardware_concurrency()));
    rich::HostMesh m;
    *mismatched = *updated = *recomputed = 0;
    for (int32_t k = 0; k < steps; k++) {
        const double *x = xs + (size_t)k * n, *y = ys + (size_t)k * n;
        rich::MeshWork work;
        work.host_edges = false;
        rich::HostMesh f;
        const int rc = rich::build_host_mesh(box, (int32_t)n, x, y, work, f, &pool);
        if (rc) return mesh_rc(rc);
        int32_t flags = 0, rounds = 0, listed = 0;
        if (k > 0 && rich::mesh_update_serial(box, (int32_t)n, x, y, m, flags, rounds, listed)) {
            *mismatched += mesh_differences(m, f);
            *updated += 1;
            *recomputed += listed;
        }
        m = std::move(f);
    }
    return RICH_OK;
}

int rich_mesh_check(rich_sim *s, int64_t *mismatched, int64_t *updates)
{
    if (!s || !mismatched) return fail(RICH_EINVAL, "bad arguments");
    if (s->pending) return fail(RICH_ESTATE, "a sweep is pending; call rich_sync first");
    if (!s->tess_current) return fail(RICH_ESTATE, "no current tessellation");
    CUDA_TRY(cudaStreamSynchronize(s->stream));
    int rc;
    rich::HostMesh d, f;
    const size_t N = (size_t)s->n, G = (size_t)s->msz.ghosts, S = (size_t)s->msz.slots;
    std::vector<double> x(N), y(N);
    auto down = [&](auto &v, const DBuf &b, size_t k) -> cudaError_t {
        v.resize(k);
        if (k == 0) return cudaSuccess;
        return cudaMemcpyAsync(v.data(), b.p, k * sizeof(v[0]), cudaMemcpyDeviceToHost, s->stream);
    };
    const int q = s->pts();
    const rich::MeshStore &m = s->mesh[s->mcur];
    CUDA_TRY(down(x, s->x[q], N)); CUDA_TRY(down(y, s->y[q], N));
    CUDA_TRY(down(d.cell_ptr, m.cell_ptr, N + 1)); CUDA_TRY(down(d.slot_nb, m.slot_nb, S));
    CUDA_TRY(down(d.tri_off, m.tri_off, N + 1)); CUDA_TRY(down(d.edge_off, m.edge_off, N + 1));
    CUDA_TRY(down(d.cell_order, m.cell_order, N));
    CUDA_TRY(down(d.gx, m.gx, G)); CUDA_TRY(down(d.gy, m.gy, G));
    CUDA_TRY(down(d.ghost_src, m.ghost_src, G)); CUDA_TRY(down(d.ghost_xf, m.ghost_xf, G));
    CUDA_TRY(down(d.ghost_shift, m.ghost_shift, G)); CUDA_TRY(down(d.ghost_img, m.ghost_img, G));
    CUDA_TRY(cudaStreamSynchronize(s->stream));
    rich::MeshWork work;
    work.host_edges = false;
    const rich::BoxConfig box{s->cfg.boundary, s->cfg.x0, s->cfg.x1, s->cfg.y0, s->cfg.y1};
    if ((rc = rich::build_host_mesh(box, s->n, x.data(), y.data(), work, f, s->pool.get()))) return mesh_rc(rc);
    *mismatched = mesh_differences(d, f);
    if (updates) *updates = s->updates;
    return RICH_OK;
}

}  // extern "C"
