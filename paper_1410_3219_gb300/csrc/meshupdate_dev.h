// Device memory and launches of the mesh update (meshupdate.h) for one set
// of cells: a simulation's, or a batch's packed ones.
#pragma once

#include "api_internal.h"
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
};

struct MeshSizes {
    int32_t ghosts = 0, tris = 0, edges = 0, slots = 0;
};

// The updated mesh (cell_ptr, slot_nb, ghost_src and ghost_img apart from
// the mesh being updated): what the host builder's upload holds.
struct MeshOutput {
    int32_t *cell_ptr, *slot_nb, *tri_off, *edge_off, *cell_order;
    double *gx, *gy;
    int32_t *ghost_src, *ghost_xf, *ghost_shift, *ghost_img;
};

class MeshUpdater {
public:
    // Enqueue the checks, the first rounds and the sizes of the updated
    // mesh, with the counters' copy to the host.
    cudaError_t start(const MeshArrays &a, cudaStream_t st);
    // After the stream was waited for: the sizes, after more rounds if
    // needed (ok = false: the rounds did not converge and the host builder
    // has to take these meshes; those of simulations with flags() too).
    cudaError_t settle(const MeshArrays &a, bool &ok, MeshSizes &sizes, cudaStream_t st);
    // Per simulation, after settle: non-zero when its mesh is left to the host.
    const int32_t *flags() const;
    // Enqueue the writing of the updated mesh.
    cudaError_t finish(const MeshArrays &a, const MeshOutput &o, cudaStream_t st);

private:
    cudaError_t reserve(int32_t n, int32_t n_inst, cudaStream_t st);
    cudaError_t read_counts(const MeshArrays &a, cudaStream_t st);
    MeshUpdate params(const MeshArrays &a) const;
    void launch_rounds(const MeshUpdate &m, int first, int last, cudaStream_t st) const;

    int32_t stamp_ = 0, max_rings_ = 0;
    DBuf mark_, list_[2], info_, at_, ring_deg_, ring_ref_, extra_n_, extra_, count_, sizes_, images_, ghost_off_,
        sums_, flags_;
    HBuf host_;
};

}  // namespace rich
