// Device memory and launches of the mesh update (meshupdate.h) for one set
// of cells: a simulation's, or a batch's packed ones.
#pragma once

#include "api_internal.h"
#include "chain.cuh"
#include "sweep.cuh"

namespace rich {

struct MeshUpdate;

// smallest and largest cell counts the update takes (below, a periodic box
// is too few spacings wide; above, references do not fit)
constexpr int32_t kMeshUpdateMin = 64, kMeshUpdateMax = 1 << 26;

// The mesh being updated and the cells' new positions (device pointers).
struct MeshArrays {
    int32_t n, n_inst;
    const InstParams *inst;    // box and mesh_params of each simulation
    const int32_t *cell_inst;  // nullptr: one simulation
    const double *x, *y;
    const int32_t *cell_ptr, *slot_nb, *ghost_src, *ghost_img;
    bool split;  // the sweep beside the update is a split-precision one
};

struct MeshSizes {
    int32_t ghosts = 0, tris = 0, edges = 0, slots = 0;
};

// The triangle and edge lists of a mesh, built on the device from its rings.
// The triangle of ring slot k of real cell i is (i, nb[k], nb[k+1]); it is
// owned by its smallest vertex id (a real cell: ghost ids follow the real
// ones), numbered in its owner's ring order from tri_off[owner] (tri_off[n] =
// T) and written rotated to start at the owner.  Real cell i owns its edges to
// larger real cells, to mirror images and (periodic box) to images of larger
// cells or of itself shifted to the +x / +y side; its owned edges are numbered
// in ring order from edge_off[i] (edge_off[n] = E).  Writes slot_edge (2 e, or
// 2 e + 1 on the partner's slot) and edge_l / edge_r / edge_ta / edge_tb
// (Voronoi edge from circumcentre ta to tb, counter-clockwise about the left
// cell), and sets *bad (and the simulation's MU_LISTS) where the rings do not
// agree with each other or with the offsets.
struct MeshLists {
    int32_t n, periodic;        // box type where cell_inst is null
    const int32_t *cell_inst;   // else each cell's box type from its simulation
    const InstParams *inst;
    const int32_t *cell_ptr, *slot_nb, *tri_off, *edge_off, *ghost_src, *ghost_shift;
    int32_t *tri, *slot_tri, *slot_edge, *edge_l, *edge_r, *edge_ta, *edge_tb;
    const uint32_t *edge_mask, *tri_mask;  // slots whose edge / triangle the cell owns (rings of up to 32), or nullptr
    const int32_t *ready;       // nullptr, or 0 there: nothing is built
    int32_t *bad;
    int32_t *flags = nullptr;   // MU_* of each simulation (an update)
    int32_t *next = nullptr, next_words = 0;  // words to clear (an update's next counters)
    // the update's counters, which the last block copies to page-locked memory
    // (`done` counts the blocks and is left at zero)
    int32_t *report = nullptr, *done = nullptr;
    const int32_t *counters = nullptr;
    int32_t words = 0;
};
// (alone: no FP64 stages run beside)
cudaError_t launch_lists(const MeshLists &l, bool alone, cudaStream_t st);

// The updated mesh (cell_ptr, slot_nb, ghost_src and ghost_img apart from
// the mesh being updated), the room its arrays have, and its lists' arrays.
struct MeshOutput {
    int32_t *cell_ptr, *slot_nb, *tri_off, *edge_off, *cell_order;
    double *gx, *gy;
    int32_t *ghost_src, *ghost_xf, *ghost_shift, *ghost_img;
    MeshSizes max;
    MeshLists lists;  // (tri .. edge_tb and periodic; the rest is filled in)
};

// The connectivity of one mesh in device memory, as host builds are uploaded
// to it and updates write it.
struct MeshStore {
    DBuf cell_ptr, slot_nb, slot_tri, slot_edge, tri, tri_off, edge_off, cell_order;
    DBuf edge_l, edge_r, edge_ta, edge_tb, gx, gy, ghost_src, ghost_xf, ghost_shift, ghost_img;
    // Room for a mesh of these sizes.  Nothing enqueued may still use the
    // arrays: those that grow are reallocated.  All are released when one fails
    // (no array has more room than another then).
    cudaError_t reserve(int32_t n, const MeshSizes &z);
    void release();
    // where an update writes, with the room there is
    MeshOutput output(int32_t periodic) const;
    // the list builder's arguments for the mesh held (its lists from its rings)
    MeshLists lists(int32_t n, int32_t periodic) const;
    // the sweep's view of it
    template <class R> void describe(SweepParams<R> &p, const MeshSizes &z) const
    {
        p.ng = z.ghosts;
        p.T = z.tris;
        p.E = z.edges;
        p.S = z.slots;
        p.gx = gx.as<double>(); p.gy = gy.as<double>();
        p.tri = tri.as<int32_t>(); p.cell_ptr = cell_ptr.as<int32_t>(); p.cell_order = cell_order.as<int32_t>();
        p.slot_nb = slot_nb.as<int32_t>(); p.slot_tri = slot_tri.as<int32_t>(); p.slot_edge = slot_edge.as<int32_t>();
        p.edge_l = edge_l.as<int32_t>(); p.edge_r = edge_r.as<int32_t>();
        p.edge_ta = edge_ta.as<int32_t>(); p.edge_tb = edge_tb.as<int32_t>();
        p.ghost_src = ghost_src.as<int32_t>(); p.ghost_xf = ghost_xf.as<int32_t>();
    }
};

// The stream that updates run on beside the rest of a sweep, and the events
// that order the two.
struct MeshStream {
    cudaStream_t stream = nullptr;
    cudaEvent_t moved = nullptr, done = nullptr;
    cudaError_t create();
    ~MeshStream();
};

struct MeshResult {
    // kDone: the mesh and its lists are written (but for the meshes of
    // simulations with flags()); kGrow: an array is too small for `sizes`;
    // kHost: no mesh is written (the only simulation is flagged, or the sizes
    // do not fit)
    enum { kDone, kGrow, kHost } state;
    MeshSizes sizes;
    bool flagged;  // some simulation's mesh is left to the host
};

class MeshUpdater {
public:
    // Enqueue the whole update, with the counters' copy to the host.  Nothing
    // is enqueued, and nothing held, when its memory cannot be had.
    cudaError_t start(const MeshArrays &a, const MeshOutput &o, cudaStream_t st);
    // After the stream was waited for: what came of it (after more rounds, if
    // the cells did not agree yet).
    cudaError_t settle(const MeshArrays &a, const MeshOutput &o, MeshResult &result, cudaStream_t st);
    // After kGrow: the mesh written to larger arrays (waits).
    cudaError_t again(const MeshArrays &a, const MeshOutput &o, MeshResult &result, cudaStream_t st);
    // Per simulation, after settle: non-zero when its mesh is left to the host.
    const int32_t *flags() const;
    // The next mesh to update is not the last update's (the host built it, or
    // the update's was not kept).
    void forget() { whole_ = true; }
    // its device memory given back (nothing enqueued may use it)
    void release();

private:
    cudaError_t reserve(int32_t n, int32_t n_inst, cudaStream_t st);
    MeshUpdate params(const MeshArrays &a, const MeshOutput &o) const;
    cudaError_t launch_rounds(const MeshArrays &a, const MeshOutput &o, int first, int last, cudaStream_t st);

    int32_t stamp_ = 0, max_rings_ = 0, last_round_ = 0;
    int quiet_ = 0;      // updates in a row that needed one round (at most kQuiet)
    bool whole_ = true;  // sizes_ does not describe the mesh to update
    bool told_ = true;   // extra_n_ may hold counts (else it is zero)
    DBuf mark_, list_[2], heavy_, info_, at_, ring_deg_, ring_ref_, extra_n_, extra_, count_[2], sizes_, images_,
        ghost_off_, sums_, edge_mask_, tri_mask_;
    HBuf host_;
};

}  // namespace rich
