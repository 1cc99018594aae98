// Batched simulations (include/rich.h, rich_batch_*): many independent
// moving-mesh simulations of different sizes and parameters advanced
// together, one device sweep per step over all of them.
//
// The simulations are packed into one index space (cells of simulation k
// follow those of k-1; ghosts, triangles, edges and ring slots likewise) with
// a per-cell simulation id and a per-simulation parameter table.  A step with
// the simulations of the last one, whose meshes the device updated, starts
// with 6; else (pack_step):
//   1. the meshes that the device updated come back to the host, and of the
//      other running simulations the points;
//   2. the simulations without a mesh, newly admitted ones included, are
//      tessellated on the host's worker threads (a0);
//   3. the meshes are packed, and the FP64 conserved state is regathered on
//      the device;
//   4. the packed meshes are uploaded;
//   5. newly admitted simulations get their conserved variables from their
//      initial primitives and first areas (geometry stage in init mode).
// Then, every step:
//   6. one sweep (a1-a9) runs over all cells; each simulation keeps its own
//      time step, remaining time and status flags; the meshes are updated for
//      the moved points (a0) beside its last stages (those of simulations
//      whose updates keep failing are built by the host meanwhile);
//   7. simulations that reached t_end or their step budget are copied out
//      and leave the batch; a failed step rolls back that simulation only;
//   8. the updated meshes become the current ones.
// The arithmetic of every cell depends only on its own simulation, so a
// simulation's results do not depend on what else is in the batch.
#include <algorithm>
#include <cstddef>
#include <cmath>
#include <cstring>
#include <limits>
#include <memory>
#include <new>
#include <string>
#include <vector>

#include "api_internal.h"
#include "mesh.h"
#include "meshupdate.h"
#include "meshupdate_dev.h"
#include "sweep.cuh"
#include "threadpool.h"

namespace {

using rich::DBuf;
using rich::now_ms;
using rich::upload;
#define CUDA_TRY RICH_CUDA_TRY

int fail(int code, const std::string &msg) { return rich::set_error(code, msg); }

enum SimState { PENDING = 0, RUNNING = 1, DONE = 2, FAILED = 3, REMOVED = 4 };

struct BatchSim {
    int32_t id = -1;
    rich_config cfg{};
    int32_t n = 0;
    std::vector<int32_t> perm;  // internal (Hilbert) -> caller index
    std::vector<double> hx, hy;  // points, internal order
    std::vector<double> W0;      // initial primitives (4n, component-major) until admitted
    rich::MeshWork mw;           // (edge lists built on the device, packed)
    rich::HostMesh hm;
    int mesh_rc = 0;
    // hm is the mesh of its current points (read back from the device, or
    // built beside the last sweep)
    bool prebuilt = false;
    int missed = 0;  // updates in a row that left its mesh to the host
    double t = 0.0, t_end = 0.0, last_dt = 0.0;
    int64_t steps = 0, max_steps = 0;
    int state = PENDING;
    int err = RICH_OK;
    std::string err_msg;
    // offsets in the packed arrays of the current step
    int64_t cell_off = -1, ghost_off = 0, tri_off = 0, edge_off = 0, slot_off = 0;
    int64_t prev_cell_off = -1;  // offset in the previous packing (-1: not packed)
    // results of a finished simulation (caller order is applied on read)
    std::vector<double> fin;  // x, y, m, px, py, E (n each, internal order)
    double t_submit = 0.0, t_admit = 0.0, t_finish = 0.0;
    BatchSim() { mw.host_edges = false; }
};

// One way of launching the sweep: stage by stage, or as one persistent
// cooperative kernel (replayed from a recorded CUDA graph) with a block size.
struct LaunchShape {
    bool persistent;
    int block;
};

int mesh_code(int rc, std::string &msg)
{
    if (rc == -2) { msg = "two generating points coincide"; return RICH_EDUPLICATE; }
    if (rc == -4) { msg = "too few points for the ghost band"; return RICH_ETOOFEW; }
    msg = "tessellation failed";
    return RICH_ETESS;
}

}  // namespace

struct rich_batch {
    int32_t precision = RICH_FP64;
    int64_t max_cells = 0;
    int64_t cells_admitted = 0;  // cells of pending + running simulations
    std::vector<std::unique_ptr<BatchSim>> sims;
    std::vector<BatchSim *> packed;  // running simulations in packed order (last step)
    int64_t n_packed = 0;            // cells in the packed arrays
    // host workers: the batch's own, or a pool it shares with other
    // batches (the server's lanes)
    std::unique_ptr<rich::ThreadPool> own_pool;
    rich::ThreadPool *pool = nullptr;
    cudaStream_t stream = nullptr;
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    // The device's mesh update (meshupdate.h) for the packed cells: after a
    // step dev_mesh says that mesh[mcur] holds the meshes of
    // the moved points of `packed` (those of simulations with a mesh flag
    // excepted), dev_lists that none is flagged and the triangle and edge
    // lists are good.  A step whose simulations are the same then starts
    // with the sweep; else the meshes are read back and packed again.
    rich::MeshUpdater updater;
    rich::MeshStore mesh[2];
    rich::MeshStream mesh_stream;
    int mcur = 0;
    bool dev_mesh = false, dev_lists = false;
    std::vector<int32_t> mesh_flag;
    // reads: the cell (within its simulation) of each caller index, packed,
    // and the state in that order: page-locked, or for a large simulation on
    // the device first
    DBuf cell_of, read_dev;
    rich::HBuf read_host;
    rich::HBuf h_back;  // dt, status per simulation, then the list builder's flag
    cudaEvent_t ev2 = nullptr, ev_read = nullptr;
    rich::HBuf h_moved;  // moved points read during a sweep: x, y (packed), then dt per simulation
    int missed = 0, host_sweeps = 0;  // as rich_sim's, of updates that failed for every simulation
    int64_t meshes_updated = 0, meshes_built = 0;  // members' meshes made on the device, and on the host
    bool diagnostics = false;
    int cur = 0;
    // device
    DBuf x[2], y[2], U[2], A, o, W, cs, g, gl, alpha, w, tess, rounding, p64, cell_inst, initW, src;
    DBuf psrc, ccx, ccy, eL, emlx, emly, emrx, emry, enx, eny, eqx, eqy, F, ePM;
    DBuf instp, dtmin, dtout, status, dsizes, gsync, listbad;
    // launch shape: autotuned over the first steps unless fixed by the caller
    int launch_mode = 0;  // 0 autotune, 1 staged, 2 persistent
    int fixed_block = 256;
    std::vector<LaunchShape> cands;
    std::vector<double> cand_ms;
    size_t cand_next = 0;
    bool tuned = false;
    LaunchShape chosen{false, 256};
    int last_grid = 0;
    bool graph_ok = true;
    std::string graph_note;
    // one recorded graph per ping-pong parity (the buffers swap roles each step)
    cudaGraph_t graph[2] = {nullptr, nullptr};
    cudaGraphExec_t gexec[2] = {nullptr, nullptr};
    std::vector<unsigned char> graph_sig[2];
    int64_t graph_records = 0;
    int64_t persistent_launches = 0, graph_launches = 0, staged_launches = 0;
    // persistent sweeps whose barrier wait gave up (each step redone staged);
    // inject_spin > 0 makes the next persistent sweep's barrier wait for one
    // block more than it launched and give up after that many polls
    int64_t barrier_timeouts = 0;
    int32_t inject_spin = 0;
    // host staging of the packed mesh
    std::vector<double> h_x, h_y, h_gx, h_gy, h_W0;
    std::vector<double> h_dlx, h_dly, h_dgx, h_dgy;  // the points (and a mesh's ghosts) downloaded at the start of a step
    std::vector<int32_t> h_dptr, h_dnb, h_dgsrc, h_dgxf, h_dgshift, h_dgimg, h_dtoff, h_deoff;
    std::vector<int32_t> h_gsrc, h_gxf, h_cell_ptr, h_slot_nb, h_cell_inst;
    std::vector<int32_t> h_corder;
    std::vector<int32_t> h_src, h_eoff, h_toff, h_gshift, h_gimg, h_cell_of;
    std::vector<rich::InstParams> h_inst;
    int64_t nG = 0, nT = 0, nE = 0, nS = 0;

    explicit rich_batch(int threads) : own_pool(new rich::ThreadPool(threads)), pool(own_pool.get()) {}
    explicit rich_batch(rich::ThreadPool *shared) : pool(shared) {}
    ~rich_batch()
    {
        if (stream) cudaStreamSynchronize(stream);
        for (int k = 0; k < 2; k++) {
            if (gexec[k]) cudaGraphExecDestroy(gexec[k]);
            if (graph[k]) cudaGraphDestroy(graph[k]);
        }
        for (cudaEvent_t e : {ev0, ev1, ev2, ev_read})
            if (e) cudaEventDestroy(e);
        if (stream) cudaStreamDestroy(stream);
    }

    double *dt_back() const { return h_back.as<double>(); }
    int32_t *status_back() const { return reinterpret_cast<int32_t *>(h_back.as<double>() + packed.size()); }
    int32_t *list_flag() const { return reinterpret_cast<int32_t *>(h_back.as<char>() + h_back.cap) - 2; }

    size_t rsize() const { return precision == RICH_FP32_SPLIT ? sizeof(float) : sizeof(double); }

    template <class R> rich::SweepParams<R> params() const
    {
        rich::SweepParams<R> p{};
        p.inst = instp.as<rich::InstParams>();
        p.cell_inst = cell_inst.as<int32_t>();
        p.n_inst = (int32_t)packed.size();
        p.diagnostics = diagnostics ? 1 : 0;
        p.motion = 1;
        p.n = (int32_t)n_packed;
        mesh[mcur].describe(p, rich::MeshSizes{(int32_t)nG, (int32_t)nT, (int32_t)nE, (int32_t)nS});
        p.x = x[cur].as<double>(); p.y = y[cur].as<double>();
        p.xn = x[1 - cur].as<double>(); p.yn = y[1 - cur].as<double>();
        p.ccx = ccx.as<double>(); p.ccy = ccy.as<double>(); p.A = A.as<double>();
        p.eL = eL.as<R>(); p.emlx = emlx.as<R>(); p.emly = emly.as<R>();
        p.emrx = emrx.as<R>(); p.emry = emry.as<R>();
        p.enx = enx.as<R>(); p.eny = eny.as<R>(); p.eqx = eqx.as<R>(); p.eqy = eqy.as<R>();
        p.ePM = ePM.as<rich::Vec4<R>>();
        p.U = U[cur].as<double>(); p.Un = U[1 - cur].as<double>();
        p.U0 = p.U; p.x0 = p.x; p.y0 = p.y;
        p.W = W.as<rich::Vec4<R>>(); p.o = o.as<rich::Vec2<R>>(); p.cs = cs.as<R>();
        p.g = g.as<rich::Vec4<R>>(); p.gl = gl.as<rich::Vec4<R>>(); p.alpha = alpha.as<rich::Vec4<R>>();
        p.w = w.as<rich::Vec2<R>>();
        p.rounding = rounding.as<uint8_t>(); p.p64 = p64.as<double>();
        p.tess = tess.as<int32_t>(); p.F = F.as<rich::Vec4<R>>(); p.psrc = psrc.as<rich::Vec4<R>>();
        p.dtmin_bits = dtmin.as<unsigned long long>();
        p.dt_out = dtout.as<double>();
        p.status = status.as<int32_t>();
        return p;
    }

    void launch(int k, const double *init_W, double *Un_override = nullptr) const
    {
        if (precision == RICH_FP32_SPLIT) {
            rich::SweepParams<float> p = params<float>();
            if (Un_override) p.Un = Un_override;
            rich::launch_stage<float>(k, p, init_W, stream);
        } else {
            rich::SweepParams<double> p = params<double>();
            if (Un_override) p.Un = Un_override;
            rich::launch_stage<double>(k, p, init_W, stream);
        }
    }

    BatchSim *find(int32_t id) const
    {
        if (id < 0 || (size_t)id >= sims.size()) return nullptr;
        BatchSim *s = sims[id].get();
        return s->state == REMOVED ? nullptr : s;
    }
};

namespace {

rich::InstParams inst_params(const BatchSim &s, bool init)
{
    rich::InstParams ip{};
    const rich_config &c = s.cfg;
    ip.gamma = c.gamma; ip.igm1 = 1.0 / (c.gamma - 1.0); ip.gamma_f = (float)ip.gamma; ip.igm1_f = (float)ip.igm1; ip.cfl = c.cfl; ip.chi = c.chi; ip.eta = c.eta; ip.theta = c.theta;
    ip.delta_v = c.delta_v; ip.delta_p = c.delta_p; ip.chi_f = (float)ip.chi; ip.theta_f = (float)ip.theta; ip.delta_v_f = (float)ip.delta_v;
    ip.x0 = c.x0; ip.x1 = c.x1; ip.y0 = c.y0; ip.y1 = c.y1;
    ip.remaining = s.t_end - s.t;
    ip.boundary = c.boundary; ip.motion = c.motion; ip.limiter = c.limiter;
    ip.init = init ? 1 : 0;
    rich::mesh_params(rich::BoxConfig{c.boundary, c.x0, c.x1, c.y0, c.y1}, s.n, ip);
    return ip;
}

// Fill the staging arrays of simulation s (index k in packing order) at its offsets.
// One piece of the packing of simulation k into the batch's index space:
// part 0 its cells [i0, i1) (points, simulation id, ring offsets, order,
// first owned edges, state sources, initial primitives), part 1 its ring
// slots [i0, i1), part 2 its triangle corners [i0, i1), part 3 its ghosts.
struct PackTask {
    int32_t k, part;
    int64_t i0, i1;
};

void pack_part(rich_batch *b, BatchSim &s, const PackTask &t)
{
    const rich::HostMesh &m = s.hm;
    const int32_t n = s.n;
    const int64_t co = s.cell_off, go = s.ghost_off, to = s.tri_off, eo = s.edge_off, so = s.slot_off;
    const int64_t N = b->n_packed;
    auto pid = [&](int32_t q) -> int32_t {
        return q < n ? (int32_t)(co + q) : (int32_t)(N + go + (q - n));
    };
    const int64_t i0 = t.i0, i1 = t.i1;
    switch (t.part) {
    case 0:
        std::memcpy(&b->h_x[co + i0], s.hx.data() + i0, sizeof(double) * (i1 - i0));
        std::memcpy(&b->h_y[co + i0], s.hy.data() + i0, sizeof(double) * (i1 - i0));
        for (int64_t i = i0; i < i1; i++) {
            b->h_cell_inst[co + i] = t.k;
            b->h_cell_of[co + s.perm[i]] = (int32_t)i;
            b->h_cell_ptr[co + i] = (int32_t)(so + m.cell_ptr[i]);
            b->h_corder[co + i] = (int32_t)(co + m.cell_order[i]);
            b->h_eoff[co + i] = (int32_t)(eo + m.edge_off[i]);
            b->h_toff[co + i] = (int32_t)(to + m.tri_off[i]);
            // conserved state: continuing simulations gather from their previous slot
            b->h_src[co + i] = s.prev_cell_off >= 0 ? (int32_t)(s.prev_cell_off + i) : -1;
        }
        if (s.state == PENDING)
            for (int c = 0; c < 4; c++)
                for (int64_t i = i0; i < i1; i++) b->h_W0[(size_t)c * N + co + i] = s.W0[(size_t)c * n + i];
        break;
    case 1:
        for (int64_t q = i0; q < i1; q++) b->h_slot_nb[so + q] = pid(m.slot_nb[q]);
        break;
    default:
        for (int64_t q = i0; q < i1; q++) {
            b->h_gx[go + q] = m.gx[q];
            b->h_gy[go + q] = m.gy[q];
            b->h_gsrc[go + q] = (int32_t)(co + m.ghost_src[q]);
            b->h_gxf[go + q] = m.ghost_xf[q];
            b->h_gshift[go + q] = m.ghost_shift[q];
            b->h_gimg[go + q] = m.ghost_img[q];
        }
        break;
    }
}

// The packing of every simulation as pieces of bounded size, so that one
// large simulation packs on all the pool's threads.
void pack_all(rich_batch *b, const std::vector<BatchSim *> &ok)
{
    constexpr int64_t kPiece = 1 << 16;
    std::vector<PackTask> tasks;
    auto split = [&](int32_t k, int32_t part, int64_t len, int64_t piece) {
        for (int64_t i = 0; i < len; i += piece) tasks.push_back(PackTask{k, part, i, std::min(len, i + piece)});
    };
    for (size_t k = 0; k < ok.size(); k++) {
        const BatchSim &s = *ok[k];
        split((int32_t)k, 0, s.n, kPiece);
        split((int32_t)k, 1, (int64_t)s.hm.slot_nb.size(), 4 * kPiece);
        split((int32_t)k, 3, s.hm.g, 4 * kPiece);
    }
    b->pool->parallel_for((int64_t)tasks.size(), [&](int64_t j) { pack_part(b, *ok[tasks[j].k], tasks[j]); });
}

int ensure_device(rich_batch *b)
{
    const size_t N = (size_t)b->n_packed, d = sizeof(double), r = b->rsize(), K = b->packed.size();
    for (int k = 0; k < 2; k++) {
        CUDA_TRY(b->x[k].ensure(N * d + 8));
        CUDA_TRY(b->y[k].ensure(N * d + 8));
    }
    // U is grown by the caller: one of its two buffers may hold the live state
    CUDA_TRY(b->A.ensure(N * d + 8)); CUDA_TRY(b->o.ensure(2 * N * r + 16));
    CUDA_TRY(b->W.ensure(4 * N * r + 32)); CUDA_TRY(b->cs.ensure(N * r + 8));
    CUDA_TRY(b->g.ensure(8 * N * r + 64)); CUDA_TRY(b->gl.ensure(8 * N * r + 64));
    CUDA_TRY(b->alpha.ensure(4 * N * r + 32)); CUDA_TRY(b->w.ensure(2 * N * r + 16));
    CUDA_TRY(b->tess.ensure(N * 4 + 4)); CUDA_TRY(b->rounding.ensure(N + 8)); CUDA_TRY(b->p64.ensure(N * d + 8));
    CUDA_TRY(b->psrc.ensure(4 * N * r + 32));
    CUDA_TRY(b->instp.ensure(K * sizeof(rich::InstParams) + 8));
    CUDA_TRY(b->dtmin.ensure(K * 8 + 8)); CUDA_TRY(b->dtout.ensure(K * 8 + 8)); CUDA_TRY(b->status.ensure(K * 4 + 8));
    CUDA_TRY(b->h_back.ensure(K * 12 + 64));
    CUDA_TRY(b->dsizes.ensure(sizeof(rich::DeviceSizes))); CUDA_TRY(b->gsync.ensure(sizeof(rich::GridSync)));
    return RICH_OK;
}

void finish_copy_out(rich_batch *b, BatchSim &s, int which)
{
    // x, y and U of simulation s from packed buffer set `which` (synchronous)
    const size_t n = (size_t)s.n, N = (size_t)b->n_packed;
    s.fin.assign(6 * n, 0.0);
    cudaMemcpyAsync(&s.fin[0], b->x[which].as<double>() + s.cell_off, n * 8, cudaMemcpyDeviceToHost, b->stream);
    cudaMemcpyAsync(&s.fin[n], b->y[which].as<double>() + s.cell_off, n * 8, cudaMemcpyDeviceToHost, b->stream);
    for (int c = 0; c < 4; c++)
        cudaMemcpyAsync(&s.fin[(2 + c) * n], b->U[which].as<double>() + c * N + s.cell_off, n * 8,
                        cudaMemcpyDeviceToHost, b->stream);
}

int sm_count()
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 1;
}

template <class R> int persistent_grid(int block)
{
    return rich::persistent_blocks_per_sm<R>(block) * sm_count();
}

// Enqueue the whole sweep as one persistent cooperative launch, from a
// recorded CUDA graph when possible.  The graph holds the barrier and status
// resets and the launch; it is recorded again only when a device buffer moved
// (the mesh sizes come from device memory).
template <class R> int run_persistent(rich_batch *b, int block)
{
    const int grid = persistent_grid<R>(block);
    if (grid <= 0) return fail(RICH_ECUDA, "persistent sweep cannot be resident");
    b->last_grid = grid;
    rich::SweepParams<R> p = b->params<R>();
    p.n = p.ng = p.T = p.E = p.S = p.n_inst = 0;  // read from device memory
    rich::DeviceSizes sz{};
    sz.n = (int32_t)b->n_packed;
    sz.ng = (int32_t)b->nG;
    sz.T = (int32_t)b->nT;
    sz.E = (int32_t)b->nE;
    sz.n_inst = (int32_t)b->packed.size();
    CUDA_TRY(cudaMemcpyAsync(b->dsizes.p, &sz, sizeof(sz), cudaMemcpyHostToDevice, b->stream));
    auto *gs = b->gsync.as<rich::GridSync>();
    auto *ds = b->dsizes.as<rich::DeviceSizes>();
    if (b->inject_spin > 0) {
        // a barrier that cannot complete: every wait runs out after
        // inject_spin polls and the sweep stops (launched directly, not from
        // the recorded graph)
        rich::GridSync g{};
        g.spin_limit = b->inject_spin;
        g.extra = 1;
        b->inject_spin = 0;
        CUDA_TRY(cudaMemcpyAsync(gs, &g, sizeof(g), cudaMemcpyHostToDevice, b->stream));
        CUDA_TRY(cudaMemsetAsync(b->status.p, 0, b->status.cap, b->stream));
        CUDA_TRY(rich::launch_persistent<R>(p, ds, gs, block, grid, b->stream));
        b->persistent_launches++;
        return RICH_OK;
    }
    if (b->graph_ok) {
        std::vector<unsigned char> sig(sizeof(p) + 3 * sizeof(int));
        std::memcpy(sig.data(), &p, sizeof(p));
        int extra[3] = {block, grid, (int)sizeof(R)};
        std::memcpy(sig.data() + sizeof(p), extra, sizeof(extra));
        const int par = b->cur;
        cudaGraph_t &graph = b->graph[par];
        cudaGraphExec_t &gexec = b->gexec[par];
        if (!gexec || sig != b->graph_sig[par]) {
            if (gexec) { cudaGraphExecDestroy(gexec); gexec = nullptr; }
            if (graph) { cudaGraphDestroy(graph); graph = nullptr; }
            bool ok = cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
            if (ok) {
                cudaMemsetAsync(gs, 0, sizeof(rich::GridSync), b->stream);
                cudaMemsetAsync(b->status.p, 0, b->status.cap, b->stream);
                cudaError_t le = rich::launch_persistent<R>(p, ds, gs, block, grid, b->stream);
                cudaError_t ce = cudaStreamEndCapture(b->stream, &graph);
                ok = le == cudaSuccess && ce == cudaSuccess && graph &&
                     cudaGraphInstantiate(&gexec, graph, 0) == cudaSuccess;
                if (!ok) b->graph_note = std::string("graph capture failed: ") + cudaGetErrorString(le != cudaSuccess ? le : ce);
            }
            cudaGetLastError();
            if (!ok) {
                b->graph_ok = false;
                if (gexec) { cudaGraphExecDestroy(gexec); gexec = nullptr; }
                if (graph) { cudaGraphDestroy(graph); graph = nullptr; }
            } else {
                b->graph_sig[par] = sig;
                b->graph_records++;
            }
        }
        if (b->graph_ok) {
            CUDA_TRY(cudaGraphLaunch(gexec, b->stream));
            b->graph_launches++;
            b->persistent_launches++;
            return RICH_OK;
        }
    }
    CUDA_TRY(cudaMemsetAsync(gs, 0, sizeof(rich::GridSync), b->stream));
    CUDA_TRY(cudaMemsetAsync(b->status.p, 0, b->status.cap, b->stream));
    CUDA_TRY(rich::launch_persistent<R>(p, ds, gs, block, grid, b->stream));
    b->persistent_launches++;
    return RICH_OK;
}

// Room for the geometry of packed meshes of these sizes (which every sweep
// computes afresh; nothing enqueued may still use the arrays).
int reserve_geometry(rich_batch *b, const rich::MeshSizes &z)
{
    const size_t T = (size_t)z.tris + 1, E = (size_t)z.edges + 1, r = b->rsize(), d = sizeof(double);
    CUDA_TRY(b->ccx.ensure(T * d)); CUDA_TRY(b->ccy.ensure(T * d));
    for (DBuf *e : {&b->eL, &b->emlx, &b->emly, &b->emrx, &b->emry, &b->enx, &b->eny, &b->eqx, &b->eqy})
        CUDA_TRY(e->ensure(E * r));
    CUDA_TRY(b->F.ensure(4 * E * sizeof(double)));
    CUDA_TRY(b->ePM.ensure(4 * E * r));
    return RICH_OK;
}

// Whether the packed cells are as many as the device's update takes.
bool fits_update(const rich_batch *b)
{
    return b->n_packed >= rich::kMeshUpdateMin && b->n_packed <= rich::kMeshUpdateMax;
}

rich::MeshArrays mesh_arrays(rich_batch *b, int q)
{
    rich::MeshArrays a{};
    a.n = (int32_t)b->n_packed;
    a.n_inst = (int32_t)b->packed.size();
    a.inst = b->instp.as<rich::InstParams>();
    a.cell_inst = b->cell_inst.as<int32_t>();
    a.x = b->x[q].as<double>();
    a.y = b->y[q].as<double>();
    const rich::MeshStore &m = b->mesh[b->mcur];
    a.cell_ptr = m.cell_ptr.as<int32_t>();
    a.slot_nb = m.slot_nb.as<int32_t>();
    a.ghost_src = m.ghost_src.as<int32_t>();
    a.ghost_img = m.ghost_img.as<int32_t>();
    a.split = b->precision == RICH_FP32_SPLIT;
    return a;
}

// Enqueue the update of the packed meshes for the points in buffers q, on the
// mesh stream from where the batch's stream is now; join_update makes the
// batch's stream continue after it.  Without memory for it nothing is enqueued,
// `update` becomes false, and the room that updates hold is given back: the
// host builds the meshes, as if every simulation's had failed before.
int start_update(rich_batch *b, int q, bool &update)
{
    rich::MeshStream &u = b->mesh_stream;
    CUDA_TRY(cudaEventRecord(u.moved, b->stream));
    CUDA_TRY(cudaStreamWaitEvent(u.stream, u.moved, 0));
    const cudaError_t e = b->updater.start(mesh_arrays(b, q), b->mesh[1 - b->mcur].output(0), u.stream);
    CUDA_TRY(rich::unless_no_room(e));
    if (e != cudaSuccess) {
        update = false;
        b->mesh[1 - b->mcur].release();
        for (BatchSim *s : b->packed) s->missed = std::max(s->missed, 2);
        b->missed = std::max(b->missed + 1, 2);
        b->host_sweeps = rich::host_sweeps_after(b->missed);
        return RICH_OK;
    }
    CUDA_TRY(cudaEventRecord(u.done, u.stream));
    return RICH_OK;
}

int join_update(rich_batch *b)
{
    CUDA_TRY(cudaStreamWaitEvent(b->stream, b->mesh_stream.done, 0));
    return RICH_OK;
}

// The moved points (in buffers q) of some simulations and the time steps to the
// host, on the mesh stream from where the batch's stream is now.
int start_read(rich_batch *b, int q, const std::vector<BatchSim *> &sims)
{
    rich::MeshStream &u = b->mesh_stream;
    const size_t N = (size_t)b->n_packed, K = b->packed.size();
    double *h = b->h_moved.as<double>();
    CUDA_TRY(cudaEventRecord(u.moved, b->stream));
    CUDA_TRY(cudaStreamWaitEvent(u.stream, u.moved, 0));
    for (const BatchSim *s : sims) {
        const size_t co = (size_t)s->cell_off, bytes = (size_t)s->n * sizeof(double);
        CUDA_TRY(cudaMemcpyAsync(h + co, b->x[q].as<double>() + co, bytes, cudaMemcpyDeviceToHost, u.stream));
        CUDA_TRY(cudaMemcpyAsync(h + N + co, b->y[q].as<double>() + co, bytes, cudaMemcpyDeviceToHost, u.stream));
    }
    CUDA_TRY(cudaMemcpyAsync(h + 2 * N, b->dtout.p, K * sizeof(double), cudaMemcpyDeviceToHost, u.stream));
    CUDA_TRY(cudaEventRecord(b->ev_read, u.stream));
    return RICH_OK;
}

// The sweep stage by stage; with `update` the mesh update for the moved points
// runs on the mesh stream beside the stages after the point motion, and the
// points of `early` are read there.
int run_staged(rich_batch *b, bool &update, const std::vector<BatchSim *> &early)
{
    CUDA_TRY(cudaMemsetAsync(b->status.p, 0, b->status.cap, b->stream));
    for (int k = 0; k < rich::NUM_STAGES; k++) {
        b->launch(k, nullptr);
        if (k != rich::K_ADVANCE) continue;
        int rc;
        if (!early.empty() && (rc = start_read(b, 1 - b->cur, early))) return rc;
        if (update && (rc = start_update(b, 1 - b->cur, update))) return rc;
    }
    CUDA_TRY(cudaGetLastError());
    b->staged_launches++;
    return RICH_OK;
}

// After the batch's stream was waited for: the meshes of the packed
// simulations on the device, as far as the update made them.
int finish_update(rich_batch *b, int q)
{
    b->dev_mesh = b->dev_lists = false;
    bool all_missed = true;
    // (a mesh made here takes the place of one that the host built meanwhile)
    auto note = [&](BatchSim *s, bool made) {
        s->missed = made ? 0 : s->missed + 1;
        if (made) s->prebuilt = false;
        if (s->state == RUNNING && made) all_missed = false;
    };
    const rich::MeshArrays a = mesh_arrays(b, q);
    rich::MeshStore &to = b->mesh[1 - b->mcur];
    cudaStream_t st = b->mesh_stream.stream;
    rich::MeshResult r;
    CUDA_TRY(b->updater.settle(a, to.output(0), r, st));
    if (r.state == rich::MeshResult::kGrow) {
        const cudaError_t e = to.reserve(a.n, r.sizes);
        CUDA_TRY(rich::unless_no_room(e));
        if (e == cudaSuccess) CUDA_TRY(b->updater.again(a, to.output(0), r, st));
    }
    const bool done = r.state == rich::MeshResult::kDone;
    for (size_t k = 0; k < b->packed.size(); k++) note(b->packed[k], done && !b->updater.flags()[k]);
    b->missed = all_missed ? b->missed + 1 : 0;
    b->host_sweeps = rich::host_sweeps_after(b->missed);
    if (!done || all_missed) {
        b->updater.forget();
        return RICH_OK;
    }
    b->mesh_flag.assign(b->updater.flags(), b->updater.flags() + a.n_inst);
    b->mcur = 1 - b->mcur;
    b->nG = r.sizes.ghosts;
    b->nT = r.sizes.tris;
    b->nE = r.sizes.edges;
    b->nS = r.sizes.slots;
    b->dev_mesh = true;
    b->dev_lists = !r.flagged;
    for (size_t k = 0; k < b->packed.size(); k++)
        b->meshes_updated += b->packed[k]->state == RUNNING && !b->mesh_flag[k];
    CUDA_TRY(rich::unless_no_room(b->mesh[1 - b->mcur].reserve(a.n, r.sizes)));
    return reserve_geometry(b, r.sizes);
}

// The meshes of the simulations that go on, read back from the device into
// their hm (with their points), for a step that packs other simulations.
int read_meshes(rich_batch *b)
{
    const size_t N = (size_t)b->n_packed, G = (size_t)b->nG, S = (size_t)b->nS;
    auto down = [&](auto &v, const DBuf &d, size_t k) -> cudaError_t {
        if (v.size() < k) v.resize(k);
        if (k == 0) return cudaSuccess;
        return cudaMemcpyAsync(v.data(), d.p, k * sizeof(v[0]), cudaMemcpyDeviceToHost, b->stream);
    };
    const rich::MeshStore &m = b->mesh[b->mcur];
    CUDA_TRY(down(b->h_dlx, b->x[b->cur], N)); CUDA_TRY(down(b->h_dly, b->y[b->cur], N));
    CUDA_TRY(down(b->h_dptr, m.cell_ptr, N + 1)); CUDA_TRY(down(b->h_dnb, m.slot_nb, S));
    CUDA_TRY(down(b->h_dtoff, m.tri_off, N + 1)); CUDA_TRY(down(b->h_deoff, m.edge_off, N + 1));
    CUDA_TRY(down(b->h_dgx, m.gx, G)); CUDA_TRY(down(b->h_dgy, m.gy, G));
    CUDA_TRY(down(b->h_dgsrc, m.ghost_src, G)); CUDA_TRY(down(b->h_dgxf, m.ghost_xf, G));
    CUDA_TRY(down(b->h_dgshift, m.ghost_shift, G)); CUDA_TRY(down(b->h_dgimg, m.ghost_img, G));
    CUDA_TRY(cudaStreamSynchronize(b->stream));
    // (ghosts follow their cells' order, so a simulation's are consecutive)
    std::vector<int64_t> g0(b->packed.size() + 1, (int64_t)G);
    for (size_t k = 0; k < b->packed.size(); k++)
        g0[k] = std::lower_bound(b->h_dgsrc.begin(), b->h_dgsrc.begin() + G, (int32_t)b->packed[k]->cell_off) -
                b->h_dgsrc.begin();
    // a window of the processing order is 1024 packed cells: it may hold
    // cells of two simulations, so each simulation's order is made again
    b->pool->parallel_for((int64_t)b->packed.size(), [&](int64_t k) {
        BatchSim *s = b->packed[k];
        if (s->state != RUNNING || b->mesh_flag[k]) return;
        const int64_t co = s->cell_off, n = s->n, go = g0[k], ge = g0[k + 1];
        rich::HostMesh &h = s->hm;
        h.n = s->n;
        h.g = (int32_t)(ge - go);
        auto slice = [&](auto &dst, const auto &src, int64_t i0, int64_t i1, int32_t shift) {
            dst.resize(i1 - i0);
            for (int64_t i = i0; i < i1; i++) dst[i - i0] = src[i] - shift;
        };
        const int32_t so = b->h_dptr[co], se = b->h_dptr[co + n];
        slice(h.cell_ptr, b->h_dptr, co, co + n + 1, so);
        slice(h.tri_off, b->h_dtoff, co, co + n + 1, b->h_dtoff[co]);
        slice(h.edge_off, b->h_deoff, co, co + n + 1, b->h_deoff[co]);
        h.n_tris = h.tri_off[n];
        h.n_edges = h.edge_off[n];
        h.slot_nb.resize(se - so);
        for (int32_t q = so; q < se; q++) {
            const int32_t id = b->h_dnb[q];
            h.slot_nb[q - so] = id < (int32_t)N ? id - (int32_t)co : (int32_t)(n + (id - (int64_t)N - go));
        }
        slice(h.gx, b->h_dgx, go, ge, 0);
        slice(h.gy, b->h_dgy, go, ge, 0);
        slice(h.ghost_src, b->h_dgsrc, go, ge, (int32_t)co);
        slice(h.ghost_xf, b->h_dgxf, go, ge, 0);
        slice(h.ghost_shift, b->h_dgshift, go, ge, 0);
        slice(h.ghost_img, b->h_dgimg, go, ge, 0);
        h.cell_order.resize(n);
        rich::degree_order((int32_t)n, h.cell_ptr.data(), h.cell_order.data());
        std::memcpy(s->hx.data(), &b->h_dlx[co], sizeof(double) * n);
        std::memcpy(s->hy.data(), &b->h_dly[co], sizeof(double) * n);
        s->mesh_rc = 0;
        s->prebuilt = true;
    });
    return RICH_OK;
}

// the launch shape of this step: the next untried candidate while tuning
LaunchShape pick_shape(rich_batch *b)
{
    if (b->launch_mode == 1) return LaunchShape{false, 256};
    if (b->launch_mode == 2) return LaunchShape{true, b->fixed_block};
    if (b->tuned) return b->chosen;
    if (b->cands.empty()) {
        // every candidate twice; the faster of its two timings counts
        for (int rep = 0; rep < 2; rep++) {
            b->cands.push_back(LaunchShape{false, 256});
            for (int bs : {128, 256, 512}) b->cands.push_back(LaunchShape{true, bs});
        }
        b->cand_ms.assign(b->cands.size(), 0.0);
    }
    return b->cands[b->cand_next];
}

void record_timing(rich_batch *b, const LaunchShape &s, double ms)
{
    if (b->launch_mode != 0 || b->tuned) return;
    b->cand_ms[b->cand_next++] = ms;
    if (b->cand_next < b->cands.size()) return;
    const size_t half = b->cands.size() / 2;
    double best = 1e300;
    for (size_t k = 0; k < half; k++) {
        double t = std::min(b->cand_ms[k], b->cand_ms[k + half]);
        if (t < best) { best = t; b->chosen = b->cands[k]; }
    }
    b->tuned = true;
    (void)s;
}

}  // namespace

namespace rich {
// A batch whose host work runs on `shared` (owned by the caller, who keeps
// it alive longer than the batch); host_threads <= 0 and shared == nullptr:
// its own pool of one thread per hardware thread.
int batch_create(int32_t precision, int64_t max_cells, int32_t host_threads, ThreadPool *shared, rich_batch **out)
{
    if (!out) return fail(RICH_EINVAL, "out is NULL");
    *out = nullptr;
    if ((precision != RICH_FP64 && precision != RICH_FP32_SPLIT) || max_cells < 3 || max_cells > ((int64_t)1 << 30))
        return fail(RICH_EINVAL, "bad precision or cell budget");
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) return fail(RICH_ENODEV, "no CUDA device");
    int threads = host_threads > 0 ? host_threads : (int)std::max(1u, std::thread::hardware_concurrency());
    rich_batch *b = shared ? new (std::nothrow) rich_batch(shared) : new (std::nothrow) rich_batch(threads);
    if (!b) return fail(RICH_ENOMEM, "host allocation");
    b->precision = precision;
    b->max_cells = max_cells;
    if (cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreate(&b->ev0) != cudaSuccess || cudaEventCreate(&b->ev1) != cudaSuccess ||
        cudaEventCreate(&b->ev2) != cudaSuccess || cudaEventCreate(&b->ev_read) != cudaSuccess ||
        b->mesh_stream.create() != cudaSuccess) {
        delete b;
        return fail(RICH_ECUDA, "stream or event creation failed");
    }
    *out = b;
    return RICH_OK;
}
}  // namespace rich

extern "C" {


int rich_batch_create(int32_t precision, int64_t max_cells, int32_t host_threads, rich_batch **out)
{
    return rich::batch_create(precision, max_cells, host_threads, nullptr, out);
}

void rich_batch_destroy(rich_batch *b) { delete b; }

int rich_batch_add(rich_batch *b, const rich_config *cfg, int64_t n, const double *x, const double *y,
                   const double *rho, const double *vx, const double *vy, const double *p, double t_end,
                   int64_t max_steps, int32_t *id)
{
    if (!b || !id) return fail(RICH_EINVAL, "NULL argument");
    if (cfg && cfg->scheme != RICH_SCHEME_EXTRAPOLATED)
        return fail(RICH_EINVAL, "batches run the extrapolated-fluxes scheme only");
    if (!rich::valid_config(cfg) || cfg->precision != b->precision)
        return fail(RICH_EINVAL, "invalid configuration or precision differs from the batch");
    if (n < 3 || n > ((int64_t)1 << 30) || !x || !y || !rho || !vx || !vy || !p) return fail(RICH_EINVAL, "bad arrays");
    if (!(t_end > 0.0) || max_steps < 1) return fail(RICH_EINVAL, "t_end must be > 0 and max_steps >= 1");
    for (int64_t i = 0; i < n; i++) {
        if (!std::isfinite(x[i]) || !std::isfinite(y[i]) || !rich::point_inside(cfg, x[i], y[i]))
            return fail(RICH_EINVAL, "point " + std::to_string(i) + " outside the box");
        if (!(rho[i] > 0) || !(p[i] > 0) || !std::isfinite(rho[i]) || !std::isfinite(p[i]) || !std::isfinite(vx[i]) ||
            !std::isfinite(vy[i]))
            return fail(RICH_EINVAL, "bad primitive values at point " + std::to_string(i));
    }
    if (b->cells_admitted + n > b->max_cells) return fail(RICH_ENOMEM, "the batch's cell budget is full");
    auto s = std::make_unique<BatchSim>();
    s->cfg = *cfg;
    s->n = (int32_t)n;
    rich::hilbert_order(s->n, x, y, s->perm);
    s->hx.resize(n);
    s->hy.resize(n);
    s->W0.resize(4 * (size_t)n);
    for (int32_t k = 0; k < s->n; k++) {
        int32_t u = s->perm[k];
        s->hx[k] = x[u];
        s->hy[k] = y[u];
        s->W0[k] = rho[u];
        s->W0[n + k] = vx[u];
        s->W0[2 * n + k] = vy[u];
        s->W0[3 * n + k] = p[u];
    }
    s->t_end = t_end;
    s->max_steps = max_steps;
    s->t_submit = now_ms();
    s->id = (int32_t)b->sims.size();  // ids index the simulation list
    *id = s->id;
    b->cells_admitted += n;
    b->sims.push_back(std::move(s));
    return RICH_OK;
}

// Simulations of at least this many cells are tessellated in tiles over the
// whole pool (four or more tiles of 16,384 points).
constexpr int32_t kTiledMember = 65536;

namespace {
// a0 for the given simulations on the pool, from the points in their hx, hy
// (results in mesh_rc): largest first, since the pool hands out tasks in
// order, so the longest tessellations start first and the makespan stays
// near the largest one (or the mean load per thread).  A simulation large
// enough for several tiles is tessellated with the whole pool (its tiles in
// parallel, as a single simulation is), one after another; the others in
// parallel, one per pool thread.  The mesh the sweep sees does not depend
// on the tiling.
void tessellate_members(rich_batch *b, const std::vector<BatchSim *> &sims)
{
    rich::Range range("rich batch tessellate (a0)");
    b->meshes_built += (int64_t)sims.size();
    std::vector<BatchSim *> by_size(sims);
    std::stable_sort(by_size.begin(), by_size.end(), [](const BatchSim *a, const BatchSim *c) { return a->n > c->n; });
    size_t n_large = 0;
    while (n_large < by_size.size() && by_size[n_large]->n >= kTiledMember) n_large++;
    for (size_t k = 0; k < n_large; k++) {
        BatchSim *s = by_size[k];
        rich::BoxConfig box{s->cfg.boundary, s->cfg.x0, s->cfg.x1, s->cfg.y0, s->cfg.y1};
        s->mesh_rc = rich::build_host_mesh(box, s->n, s->hx.data(), s->hy.data(), s->mw, s->hm, b->pool);
    }
    b->pool->parallel_for((int64_t)(by_size.size() - n_large), [&](int64_t k) {
        BatchSim *s = by_size[n_large + k];
        rich::BoxConfig box{s->cfg.boundary, s->cfg.x0, s->cfg.x1, s->cfg.y0, s->cfg.y1};
        s->mesh_rc = rich::build_host_mesh(box, s->n, s->hx.data(), s->hy.data(), s->mw, s->hm);
    });
}

// Steps 1 to 5 of a step whose meshes are not all on the device: the points
// and meshes of `list` on the host, packed, uploaded, and new simulations
// initialised.  t1, t2: when the host tessellations began and ended.
int pack_step(rich_batch *b, const std::vector<BatchSim *> &list, double &t1, double &t2)
{
    // 1. the meshes the device updated, and the points of the other running
    //    simulations, back to the host
    int rc;
    if (b->dev_mesh && (rc = read_meshes(b))) return rc;
    b->dev_mesh = b->dev_lists = false;
    bool need_points = false;
    for (BatchSim *s : b->packed) need_points |= s->state == RUNNING && !s->prebuilt;
    if (b->n_packed > 0 && need_points) {
        // (kept between steps: a fresh vector would zero 16 B per cell first)
        std::vector<double> &hx = b->h_dlx, &hy = b->h_dly;
        if (hx.size() < (size_t)b->n_packed) {
            hx.resize(b->n_packed);
            hy.resize(b->n_packed);
        }
        CUDA_TRY(cudaMemcpyAsync(hx.data(), b->x[b->cur].p, b->n_packed * 8, cudaMemcpyDeviceToHost, b->stream));
        CUDA_TRY(cudaMemcpyAsync(hy.data(), b->y[b->cur].p, b->n_packed * 8, cudaMemcpyDeviceToHost, b->stream));
        CUDA_TRY(cudaStreamSynchronize(b->stream));
        // to each simulation's own arrays, on the pool
        b->pool->parallel_for((int64_t)b->packed.size(), [&](int64_t k) {
            BatchSim *s = b->packed[k];
            if (s->state != RUNNING || s->prebuilt) return;
            std::memcpy(s->hx.data(), &hx[s->cell_off], sizeof(double) * s->n);
            std::memcpy(s->hy.data(), &hy[s->cell_off], sizeof(double) * s->n);
        });
    }
    for (BatchSim *s : list) s->prev_cell_off = s->state == RUNNING ? s->cell_off : -1;
    // 2. tessellations in parallel (of the simulations whose mesh the device
    //    did not have)
    t1 = now_ms();
    {
        std::vector<BatchSim *> todo;
        for (BatchSim *s : list)
            if (!s->prebuilt) todo.push_back(s);
        tessellate_members(b, todo);
        for (BatchSim *s : list) s->prebuilt = false;
    }
    t2 = now_ms();
    std::vector<BatchSim *> ok;
    for (BatchSim *s : list) {
        if (s->mesh_rc == 0) {
            ok.push_back(s);
            continue;
        }
        s->err = mesh_code(s->mesh_rc, s->err_msg);
        if (s->state == RUNNING) {
            // keep its last good state for the caller
            s->cell_off = s->prev_cell_off;
            finish_copy_out(b, *s, b->cur);
        }
        s->state = FAILED;
        s->t_finish = now_ms();
        b->cells_admitted -= s->n;
    }
    CUDA_TRY(cudaStreamSynchronize(b->stream));
    // 3. packing offsets
    const int64_t n_old = b->n_packed;
    bool same_layout = ok.size() == b->packed.size();
    int64_t co = 0, go = 0, to = 0, eo = 0, so = 0;
    for (size_t k = 0; k < ok.size(); k++) {
        BatchSim *s = ok[k];
        if (same_layout && (b->packed[k] != s || s->prev_cell_off != co)) same_layout = false;
        s->cell_off = co; s->ghost_off = go; s->tri_off = to; s->edge_off = eo; s->slot_off = so;
        co += s->n;
        go += s->hm.g;
        to += (int64_t)s->hm.n_tris;
        eo += (int64_t)s->hm.n_edges;
        so += (int64_t)s->hm.slot_nb.size();
    }
    if (co + go > ((int64_t)1 << 31) - 1 || 3 * to > ((int64_t)1 << 31) - 1 || 2 * eo > ((int64_t)1 << 31) - 1)
        return fail(RICH_ENOMEM, "batch exceeds 32-bit indexing");
    b->packed = ok;
    b->n_packed = co;
    b->nG = go;
    b->nT = to;
    b->nE = eo;
    b->nS = so;
    const size_t N = (size_t)co;
    bool any_pending = false;
    for (BatchSim *s : ok) any_pending |= s->state == PENDING;
    b->h_x.resize(N); b->h_y.resize(N); b->h_cell_inst.resize(N); b->h_src.resize(N);
    b->h_cell_of.resize(N);
    b->h_gx.resize(go); b->h_gy.resize(go); b->h_gsrc.resize(go); b->h_gxf.resize(go);
    b->h_cell_ptr.resize(N + 1); b->h_corder.resize(N);
    b->h_slot_nb.resize(so);
    b->h_eoff.resize(N + 1); b->h_toff.resize(N + 1); b->h_gshift.resize(go);
    b->h_gimg.resize(go);
    if (any_pending) b->h_W0.assign(4 * N, 0.0);
    pack_all(b, ok);
    b->h_cell_ptr[N] = (int32_t)so;
    b->h_eoff[N] = (int32_t)eo;
    b->h_toff[N] = (int32_t)to;
    b->h_inst.resize(ok.size());
    for (size_t k = 0; k < ok.size(); k++) b->h_inst[k] = inst_params(*ok[k], ok[k]->state == PENDING);
    // 4. device buffers and uploads
    if ((rc = ensure_device(b))) return rc;
    const rich::MeshSizes z{(int32_t)go, (int32_t)to, (int32_t)eo, (int32_t)so};
    b->updater.forget();
    CUDA_TRY(b->mesh[b->mcur].reserve((int32_t)N, z));
    if ((rc = reserve_geometry(b, z))) return rc;
    // (the other store too where an update follows, as far as there is memory)
    if (fits_update(b) && b->host_sweeps == 0)
        CUDA_TRY(rich::unless_no_room(b->mesh[1 - b->mcur].reserve((int32_t)N, z)));
    const int nxt = 1 - b->cur;
    if (!same_layout && n_old > 0) {
        // regather the conserved state of continuing simulations into the other
        // buffer (grown first: U[cur] holds the live state and is not touched)
        CUDA_TRY(b->U[nxt].ensure(4 * N * sizeof(double) + 8));
        CUDA_TRY(upload(b->src, b->h_src, b->stream));
        rich::launch_repack(b->src.as<int32_t>(), (int32_t)N, (int32_t)n_old, b->U[b->cur].as<double>(),
                            b->U[nxt].as<double>(), b->stream);
        CUDA_TRY(cudaGetLastError());
        b->cur = nxt;
    } else if (n_old == 0) {
        CUDA_TRY(b->U[b->cur].ensure(4 * N * sizeof(double) + 8));  // nothing live yet
    }
    // the buffer the sweep writes; its old contents are dead
    CUDA_TRY(cudaStreamSynchronize(b->stream));
    CUDA_TRY(b->U[1 - b->cur].ensure(4 * N * sizeof(double) + 8));
    CUDA_TRY(upload(b->x[b->cur], b->h_x, b->stream));
    CUDA_TRY(upload(b->y[b->cur], b->h_y, b->stream));
    CUDA_TRY(upload(b->cell_inst, b->h_cell_inst, b->stream));
    CUDA_TRY(upload(b->cell_of, b->h_cell_of, b->stream));
    rich::MeshStore &d = b->mesh[b->mcur];
    CUDA_TRY(upload(d.gx, b->h_gx, b->stream));
    CUDA_TRY(upload(d.gy, b->h_gy, b->stream));
    CUDA_TRY(upload(d.ghost_src, b->h_gsrc, b->stream));
    CUDA_TRY(upload(d.ghost_img, b->h_gimg, b->stream));
    CUDA_TRY(upload(d.ghost_xf, b->h_gxf, b->stream));
    CUDA_TRY(upload(d.ghost_shift, b->h_gshift, b->stream));
    CUDA_TRY(upload(d.cell_ptr, b->h_cell_ptr, b->stream));
    CUDA_TRY(upload(d.cell_order, b->h_corder, b->stream));
    CUDA_TRY(upload(d.slot_nb, b->h_slot_nb, b->stream));
    CUDA_TRY(upload(d.tri_off, b->h_toff, b->stream));
    CUDA_TRY(upload(d.edge_off, b->h_eoff, b->stream));
    CUDA_TRY(upload(b->instp, b->h_inst, b->stream));
    // the packed triangle and edge lists, checked before any kernel reads them
    {
        CUDA_TRY(b->listbad.ensure(8));
        rich::MeshLists l = d.lists((int32_t)N, 0);
        l.cell_inst = b->cell_inst.as<int32_t>();
        l.inst = b->instp.as<rich::InstParams>();
        l.bad = b->listbad.as<int32_t>();
        CUDA_TRY(cudaMemsetAsync(l.bad, 0, 4, b->stream));
        CUDA_TRY(rich::launch_lists(l, true, b->stream));
        CUDA_TRY(cudaMemcpyAsync(b->list_flag(), l.bad, 4, cudaMemcpyDeviceToHost, b->stream));
        CUDA_TRY(cudaStreamSynchronize(b->stream));
        if (*b->list_flag()) return fail(RICH_ETESS, "the rings of a mesh do not close");
    }
    CUDA_TRY(cudaMemsetAsync(b->status.p, 0, ok.size() * 4, b->stream));
    if (any_pending) CUDA_TRY(upload(b->initW, b->h_W0, b->stream));
    // 5. admission: conserved variables of new simulations from their first geometry
    if (any_pending) {
        b->launch(rich::K_CIRCUMCENTRE, nullptr);
        b->launch(rich::K_GEOMETRY, b->initW.as<double>(), b->U[b->cur].as<double>());
        for (BatchSim *s : ok)
            if (s->state == PENDING) {
                s->state = RUNNING;
                s->t_admit = now_ms();
                s->W0.clear();
                s->W0.shrink_to_fit();
            }
        for (size_t k = 0; k < ok.size(); k++) b->h_inst[k].init = 0;
        CUDA_TRY(upload(b->instp, b->h_inst, b->stream));
    }
    return RICH_OK;
}

}  // namespace

int rich_batch_step(rich_batch *b, rich_step_info *info)
{
    rich::Range range("rich batch step");
    if (!b) return fail(RICH_EINVAL, "NULL handle");
    if (info) std::memset(info, 0, sizeof(*info));
    const double t0 = now_ms();
    // the simulations of this step: running ones in their previous order, then new ones
    std::vector<BatchSim *> list;
    for (BatchSim *s : b->packed)
        if (s->state == RUNNING) list.push_back(s);
    for (auto &s : b->sims)
        if (s->state == PENDING) list.push_back(s.get());
    if (list.empty()) {
        b->packed.clear();
        b->n_packed = 0;
        b->dev_mesh = b->dev_lists = false;
        return RICH_OK;
    }
    int rc;
    double t1 = now_ms(), t2 = t1;
    if (b->dev_lists && list == b->packed) {
        // their meshes, lists and points are on the device already
        for (size_t k = 0; k < list.size(); k++) b->h_inst[k] = inst_params(*list[k], false);
        b->dev_mesh = b->dev_lists = false;
        CUDA_TRY(upload(b->instp, b->h_inst, b->stream));
    } else if ((rc = pack_step(b, list, t1, t2))) {
        return rc;
    }
    if (b->packed.empty()) return RICH_OK;
    const double t3 = now_ms();
    // 6. the sweep over every cell of every simulation, and the mesh update for
    //    the moved points (staged: beside the last stages; one wait for both)
    const std::vector<BatchSim *> ok = b->packed;
    const size_t N = (size_t)b->n_packed;
    // (static meshes' points stay where they are, bit for bit: x + dt 0)
    bool still = true;
    for (const BatchSim *s : ok) still = still && s->cfg.motion == RICH_MESH_EULERIAN;
    const bool fits = fits_update(b);
    const LaunchShape shape = pick_shape(b);
    // simulations whose meshes the host builds while a staged sweep ends: those
    // that the last two updates could not make (they are tried again with the
    // others', or now and then where there are no others)
    std::vector<BatchSim *> early;
    bool hopeful = false;
    for (BatchSim *s : ok) {
        const bool wait = s->missed >= 2;
        hopeful = hopeful || !wait;
        if (!still && !shape.persistent && (wait || !fits)) early.push_back(s);
    }
    bool update = !still && fits && (hopeful || b->host_sweeps == 0);
    if (!still && fits && !update) b->host_sweeps--;
    if (!early.empty()) CUDA_TRY(b->h_moved.ensure((2 * N + ok.size()) * sizeof(double)));
    CUDA_TRY(cudaEventRecord(b->ev0, b->stream));
    if (shape.persistent) {
        rc = b->precision == RICH_FP32_SPLIT ? run_persistent<float>(b, shape.block) : run_persistent<double>(b, shape.block);
    } else {
        rc = run_staged(b, update, early);
    }
    if (rc) return rc;
    CUDA_TRY(cudaEventRecord(b->ev1, b->stream));
    if (shape.persistent) {
        int32_t timeout = 0;
        CUDA_TRY(cudaMemcpyAsync(&timeout, (char *)b->gsync.p + offsetof(rich::GridSync, timeout), 4,
                                 cudaMemcpyDeviceToHost, b->stream));
        CUDA_TRY(cudaStreamSynchronize(b->stream));
        if (timeout) {
            // a barrier wait gave up: the inputs of the step are untouched, so
            // redo it stage by stage and keep the staged launch from now on
            b->launch_mode = 1;
            b->barrier_timeouts++;
            b->graph_note = "persistent sweep barrier timed out; staged launches used";
            CUDA_TRY(cudaEventRecord(b->ev0, b->stream));
            bool none = false;
            if ((rc = run_staged(b, none, {}))) return rc;
            CUDA_TRY(cudaEventRecord(b->ev1, b->stream));
        }
    }
    if (update && shape.persistent && (rc = start_update(b, 1 - b->cur, update))) return rc;
    // (copied while the update still runs)
    CUDA_TRY(cudaMemcpyAsync(b->dt_back(), b->dtout.p, ok.size() * 8, cudaMemcpyDeviceToHost, b->stream));
    CUDA_TRY(cudaMemcpyAsync(b->status_back(), b->status.p, ok.size() * 4, cudaMemcpyDeviceToHost, b->stream));
    if (update && (rc = join_update(b))) return rc;
    CUDA_TRY(cudaEventRecord(b->ev2, b->stream));
    double t_pre = 0.0;
    if (!early.empty()) {
        CUDA_TRY(cudaEventSynchronize(b->ev_read));
        const double tp = now_ms();
        const double *h = b->h_moved.as<double>();
        // those that go on after this step (the bookkeeping below takes the
        // same decision), unless the step fails
        std::vector<BatchSim *> next;
        for (size_t k = 0, e = 0; k < ok.size() && e < early.size(); k++) {
            BatchSim *s = ok[k];
            if (s != early[e]) continue;
            e++;
            const double dt = h[2 * N + k], rem = s->t_end - s->t;
            const double tn = dt >= rem ? s->t_end : s->t + dt;
            if (tn >= s->t_end || s->steps + 1 >= s->max_steps) continue;
            next.push_back(s);
        }
        b->pool->parallel_for((int64_t)next.size(), [&](int64_t k) {
            BatchSim *s = next[k];
            std::memcpy(s->hx.data(), h + s->cell_off, sizeof(double) * s->n);
            std::memcpy(s->hy.data(), h + N + s->cell_off, sizeof(double) * s->n);
        });
        tessellate_members(b, next);
        for (BatchSim *s : next) s->prebuilt = true;
        t_pre = now_ms() - tp;
    }
    CUDA_TRY(cudaStreamSynchronize(b->stream));
    float ms = 0.0f;
    cudaEventElapsedTime(&ms, b->ev0, b->ev1);
    // (what the update takes beyond the end of the sweep; the launch shapes are
    // compared by the whole)
    float up_ms = 0.0f;
    cudaEventElapsedTime(&up_ms, b->ev1, b->ev2);
    record_timing(b, shape, ms + up_ms);
    // 7. per-simulation bookkeeping; a failed step keeps that simulation's old state
    const int nxt2 = 1 - b->cur;
    const double tnow = now_ms();
    const int32_t *status = b->status_back();
    size_t going = 0;
    for (size_t k = 0; k < ok.size(); k++) {
        BatchSim *s = ok[k];
        if (status[k]) {
            s->prebuilt = false;
            s->err = (status[k] & rich::ST_NAN) ? RICH_ENAN : RICH_ENEGATIVE;
            s->err_msg = "step rejected (non-finite, non-positive mass or thermal energy, or a point left the box)";
            finish_copy_out(b, *s, b->cur);
            s->state = FAILED;
            s->t_finish = tnow;
            b->cells_admitted -= s->n;
            continue;
        }
        const double rem = s->t_end - s->t;
        s->last_dt = b->dt_back()[k];
        s->t = s->last_dt >= rem ? s->t_end : s->t + s->last_dt;
        s->steps++;
        if (s->t >= s->t_end || s->steps >= s->max_steps) {
            finish_copy_out(b, *s, nxt2);
            s->state = DONE;
            s->t_finish = tnow;
            b->cells_admitted -= s->n;
        } else {
            going++;
        }
    }
    if (going < ok.size()) CUDA_TRY(cudaStreamSynchronize(b->stream));
    b->cur = nxt2;
    // 8. the updated meshes of the simulations that go on
    const double tf = now_ms();
    if (update && going > 0 && (rc = finish_update(b, nxt2))) return rc;
    if (update && going == 0) b->updater.forget();
    if (still && going > 0) {
        b->mesh_flag.assign(ok.size(), 0);
        b->dev_mesh = b->dev_lists = true;
    }
    const double t_fin = now_ms() - tf;
    if (info) {
        info->steps_done = (int64_t)ok.size();
        info->sweep_ms = ms;
        info->tess_ms = (t2 - t1) + t_pre + up_ms + t_fin;
        info->copy_ms = (t1 - t0) + (t3 - t2) + (now_ms() - tnow) - t_fin;
        info->n_ghost = b->nG;
        info->n_tri = b->nT;
        info->n_edges = b->nE;
        info->n_slots = b->nS;
        info->t = 0.0;
        info->dt_last = 0.0;
    }
    return RICH_OK;
}

int rich_batch_query(rich_batch *b, int32_t id, int32_t *state, int32_t *error, double *t, int64_t *steps,
                     double *latency_ms)
{
    if (!b) return fail(RICH_EINVAL, "NULL handle");
    BatchSim *s = b->find(id);
    if (!s) return fail(RICH_EINVAL, "unknown simulation id");
    if (state) *state = s->state;
    if (error) *error = s->err;
    if (t) *t = s->t;
    if (steps) *steps = s->steps;
    if (latency_ms)
        *latency_ms = (s->state == DONE || s->state == FAILED) ? s->t_finish - s->t_submit : -1.0;
    return RICH_OK;
}

int rich_batch_get_conserved(rich_batch *b, int32_t id, int64_t n, double *x, double *y, double *m, double *px,
                             double *py, double *E)
{
    if (!b) return fail(RICH_EINVAL, "NULL handle");
    BatchSim *s = b->find(id);
    if (!s || n != s->n) return fail(RICH_EINVAL, "unknown simulation id or wrong size");
    double *outs[6] = {x, y, m, px, py, E};
    if (s->state == DONE || s->state == FAILED) {
        if (s->fin.empty()) return fail(RICH_ESTATE, "no state recorded");
        const double *src = s->fin.data();
        for (int f = 0; f < 6; f++) {
            if (!outs[f]) continue;
            for (int32_t k = 0; k < s->n; k++) outs[f][s->perm[k]] = src[(size_t)f * s->n + k];
        }
    } else if (s->state == RUNNING) {
        // put in the caller's order on the device, straight into page-locked
        // memory (24 us for 4,096 cells, 28 by one copy; 111 and 118 for 32,761)
        // or, where a gather at the link's pace would hold the SMs that other
        // batches' sweeps use for long, by one copy (65,536 cells: 242 us, 215
        // straight; 160,000: 570 and 530).  Without memory for that the host
        // reorders.
        const size_t nn = (size_t)s->n, N = (size_t)b->n_packed, co = (size_t)s->cell_off;
        const double *U = b->U[b->cur].as<double>() + co;
        const double *src[6] = {b->x[b->cur].as<double>() + co, b->y[b->cur].as<double>() + co, U, U + N, U + 2 * N,
                                U + 3 * N};
        const bool direct = 6 * nn * 8 <= ((size_t)2 << 20);
        CUDA_TRY(rich::unless_no_room(b->read_host.ensure(6 * nn * 8)));
        if (!direct) CUDA_TRY(rich::unless_no_room(b->read_dev.ensure(6 * nn * 8)));
        if (!b->read_host.p || (!direct && !b->read_dev.p)) {
            std::vector<double> h(nn);
            for (int f = 0; f < 6; f++) {
                if (!outs[f]) continue;
                CUDA_TRY(cudaMemcpyAsync(h.data(), src[f], nn * 8, cudaMemcpyDeviceToHost, b->stream));
                CUDA_TRY(cudaStreamSynchronize(b->stream));
                for (size_t k = 0; k < nn; k++) outs[f][s->perm[k]] = h[k];
            }
            return RICH_OK;
        }
        double *to = direct ? b->read_host.as<double>() : b->read_dev.as<double>();
        CUDA_TRY(rich::launch_unpermute(s->n, b->cell_of.as<int32_t>() + co, src, to, b->stream));
        if (!direct) CUDA_TRY(cudaMemcpyAsync(b->read_host.p, to, 6 * nn * 8, cudaMemcpyDeviceToHost, b->stream));
        CUDA_TRY(cudaStreamSynchronize(b->stream));
        for (int f = 0; f < 6; f++)
            if (outs[f]) std::memcpy(outs[f], b->read_host.as<double>() + (size_t)f * nn, nn * 8);
    } else {
        return fail(RICH_ESTATE, "simulation not admitted yet");
    }
    return RICH_OK;
}

int rich_batch_remove(rich_batch *b, int32_t id)
{
    if (!b) return fail(RICH_EINVAL, "NULL handle");
    BatchSim *s = b->find(id);
    if (!s) return fail(RICH_EINVAL, "unknown simulation id");
    if (s->state == PENDING || s->state == RUNNING) b->cells_admitted -= s->n;
    s->state = REMOVED;
    s->fin.clear();
    s->fin.shrink_to_fit();
    s->hm = rich::HostMesh();
    s->mw = rich::MeshWork();
    s->hx = std::vector<double>();
    s->hy = std::vector<double>();
    s->perm = std::vector<int32_t>();
    s->W0 = std::vector<double>();
    return RICH_OK;
}

int rich_batch_set_diagnostics(rich_batch *b, int32_t on)
{
    if (!b) return fail(RICH_EINVAL, "NULL handle");
    b->diagnostics = on != 0;
    return RICH_OK;
}

int64_t rich_batch_cells(const rich_batch *b) { return b ? b->cells_admitted : -1; }

int rich_batch_set_launch(rich_batch *b, int32_t mode, int32_t block)
{
    if (!b) return fail(RICH_EINVAL, "NULL handle");
    if (mode < 0 || mode > 2 || (mode == 2 && block != 128 && block != 256 && block != 512))
        return fail(RICH_EINVAL, "mode 0 (autotune), 1 (staged) or 2 (persistent, block 128/256/512)");
    b->launch_mode = mode;
    b->fixed_block = block;
    b->tuned = false;
    b->cands.clear();
    b->cand_next = 0;
    return RICH_OK;
}

int rich_batch_mesh_counts(const rich_batch *b, int64_t *updated, int64_t *built)
{
    if (!b || !updated || !built) return fail(RICH_EINVAL, "bad arguments");
    *updated = b->meshes_updated;
    *built = b->meshes_built;
    return RICH_OK;
}

int rich_batch_inject_barrier_timeout(rich_batch *b, int32_t spin_limit, int64_t *timeouts_seen)
{
    if (!b || spin_limit < 0) return fail(RICH_EINVAL, "bad arguments");
    if (spin_limit > 0) b->inject_spin = spin_limit;
    if (timeouts_seen) *timeouts_seen = b->barrier_timeouts;
    return RICH_OK;
}

int rich_batch_launch_info(const rich_batch *b, int32_t *persistent, int32_t *block, int32_t *grid, int32_t *tuned,
                           int32_t *graph, int64_t *counts)
{
    if (!b) return fail(RICH_EINVAL, "NULL handle");
    LaunchShape s = b->launch_mode == 1 ? LaunchShape{false, 256}
                    : b->launch_mode == 2 ? LaunchShape{true, b->fixed_block}
                                          : b->chosen;
    if (persistent) *persistent = s.persistent ? 1 : 0;
    if (block) *block = s.block;
    if (grid) *grid = b->last_grid;
    if (tuned) *tuned = (b->launch_mode != 0 || b->tuned) ? 1 : 0;
    if (graph) *graph = b->graph_ok ? 1 : 0;
    if (counts) {
        counts[0] = b->staged_launches;
        counts[1] = b->persistent_launches;
        counts[2] = b->graph_launches;
        counts[3] = b->graph_records;
    }
    return RICH_OK;
}

}  // extern "C"
