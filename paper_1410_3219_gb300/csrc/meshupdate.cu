// Kernels of the mesh update (bodies and method: meshupdate.h) and the class
// that holds its device memory.  Compiled without floating-point contraction
// (the predicates' error bounds assume it).
#include "meshupdate_dev.h"

#include <algorithm>

#include "meshupdate.h"

namespace rich {
namespace {

constexpr int kVerifyBlock = 128;
constexpr int kListBlock = 64;
constexpr int kWindow = kOrderWindow;  // cells per block of the size and ring passes
static_assert(kWindow == 1024, "the scans and the order pass run one window per 1024-thread block");

__global__ void __launch_bounds__(kVerifyBlock) k_mesh_verify(MeshUpdate m)
{
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < m.n) mu::verify(m, i);
}

__global__ void __launch_bounds__(kListBlock) k_mesh_recompute(MeshUpdate m, int32_t round)
{
    const int32_t count = m.count->listed[round];
    for (int32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < count; k += gridDim.x * blockDim.x)
        mu::recompute(m, m.list[round & 1][k], round);
}

__global__ void __launch_bounds__(kListBlock) k_mesh_check(MeshUpdate m, int32_t round)
{
    const int32_t count = m.count->listed[round];
    for (int32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < count; k += gridDim.x * blockDim.x)
        mu::check(m, m.list[round & 1][k], round);
}

__device__ __forceinline__ int4 plus(int4 a, int4 b) { return make_int4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }

// inclusive sum over the block's 1024 threads
__device__ __forceinline__ int4 block_sum(int4 v, int4 *warp_sums)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int o = 1; o < 32; o <<= 1) {
        int4 u;
        u.x = __shfl_up_sync(0xffffffffu, v.x, o);
        u.y = __shfl_up_sync(0xffffffffu, v.y, o);
        u.z = __shfl_up_sync(0xffffffffu, v.z, o);
        u.w = __shfl_up_sync(0xffffffffu, v.w, o);
        if (lane >= o) v = plus(v, u);
    }
    if (lane == 31) warp_sums[wid] = v;
    __syncthreads();
    if (wid == 0) {
        int4 w = warp_sums[lane];
        for (int o = 1; o < 32; o <<= 1) {
            int4 u;
            u.x = __shfl_up_sync(0xffffffffu, w.x, o);
            u.y = __shfl_up_sync(0xffffffffu, w.y, o);
            u.z = __shfl_up_sync(0xffffffffu, w.z, o);
            u.w = __shfl_up_sync(0xffffffffu, w.w, o);
            if (lane >= o) w = plus(w, u);
        }
        warp_sums[lane] = w;
    }
    __syncthreads();
    return wid ? plus(v, warp_sums[wid - 1]) : v;
}

__device__ __forceinline__ int4 sizes_of(uint32_t s)
{
    return make_int4((int)(s & 255), (int)(s >> 8 & 255), (int)(s >> 16 & 255), (int)(s >> 24));
}

// sizes per cell and their sums per window
__global__ void __launch_bounds__(kWindow) k_mesh_measure(MeshUpdate m, int4 *window_sums)
{
    __shared__ int4 ws[32];
    const int32_t i = blockIdx.x * kWindow + threadIdx.x;
    const int4 v = block_sum(i < m.n ? sizes_of(mu::measure(m, i)) : make_int4(0, 0, 0, 0), ws);
    if (threadIdx.x == kWindow - 1) window_sums[blockIdx.x] = v;
}

// window sums -> the sums before each window, and the totals
__global__ void __launch_bounds__(kWindow) k_mesh_totals(MeshUpdate m, int4 *window_sums, int32_t windows)
{
    __shared__ int4 ws[32];
    __shared__ int4 carry;
    if (threadIdx.x == 0) carry = make_int4(0, 0, 0, 0);
    __syncthreads();
    for (int32_t base = 0; base < windows; base += kWindow) {
        const int32_t k = base + threadIdx.x;
        const int4 own = k < windows ? window_sums[k] : make_int4(0, 0, 0, 0);
        const int4 inc = block_sum(own, ws);
        const int4 c = carry;
        if (k < windows)
            window_sums[k] = make_int4(c.x + inc.x - own.x, c.y + inc.y - own.y, c.z + inc.z - own.z, c.w + inc.w - own.w);
        __syncthreads();
        if (threadIdx.x == kWindow - 1) carry = plus(c, inc);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        m.count->slots = carry.x;
        m.count->edges = carry.y;
        m.count->tris = carry.z;
        m.count->ghosts = carry.w;
    }
}

// offsets per cell, the ghosts, and the processing order: within each window
// cells by decreasing ring degree, stable (degree_order in mesh.cpp)
__global__ void __launch_bounds__(kWindow) k_mesh_offsets(MeshUpdate m, const int4 *window_sums, int32_t *order)
{
    __shared__ int4 ws[32];
    __shared__ int32_t hist[32][65];  // cells of each degree in each warp, then their first places
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int32_t i = blockIdx.x * kWindow + threadIdx.x;
    const int4 own = i < m.n ? sizes_of(m.sizes[i]) : make_int4(0, 0, 0, 0);
    const int4 inc = block_sum(own, ws), base = window_sums[blockIdx.x];
    const int4 at = make_int4(base.x + inc.x - own.x, base.y + inc.y - own.y, base.z + inc.z - own.z,
                              base.w + inc.w - own.w);
    if (i < m.n) {
        m.out_ptr[i] = at.x;
        m.edge_off[i] = at.y;
        m.tri_off[i] = at.z;
        m.ghost_off[i] = at.w;
        if (i == m.n - 1) {
            m.out_ptr[m.n] = at.x + own.x;
            m.edge_off[m.n] = at.y + own.y;
            m.tri_off[m.n] = at.z + own.z;
            m.ghost_off[m.n] = at.w + own.w;
        }
        mu::place_ghosts(m, i);
    }
    for (int k = threadIdx.x; k < 32 * 65; k += kWindow) (&hist[0][0])[k] = 0;
    __syncthreads();
    const int deg = i < m.n ? (own.x < 64 ? own.x : 64) : -1;
    const unsigned same = __match_any_sync(0xffffffffu, deg);
    const int before = __popc(same & ((1u << lane) - 1));
    if (deg >= 0 && before == 0) hist[wid][deg] = __popc(same);
    __syncthreads();
    if (threadIdx.x < 65) {
        int run = 0;
        for (int w = 0; w < 32; w++) {
            const int c = hist[w][threadIdx.x];
            hist[w][threadIdx.x] = run;
            run += c;
        }
        ((int *)ws)[threadIdx.x] = run;  // cells of this degree in the window (65 ints in 128)
    }
    __syncthreads();
    if (deg >= 0) {
        int place = hist[wid][deg] + before;
        for (int d = deg + 1; d <= 64; d++) place += ((int *)ws)[d];
        order[blockIdx.x * kWindow + place] = i;
    }
}

__global__ void __launch_bounds__(256) k_mesh_rings(MeshUpdate m)
{
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < m.n) mu::place_ring(m, i);
}

inline int blocks(int64_t n, int b) { return (int)((n + b - 1) / b); }

}  // namespace

#define MU_TRY(e)                               \
    do {                                        \
        const cudaError_t err_ = (e);           \
        if (err_ != cudaSuccess) return err_;   \
    } while (0)

cudaError_t MeshUpdater::reserve(int32_t n, int32_t n_inst, cudaStream_t st)
{
    const size_t N = (size_t)n, i4 = sizeof(int32_t);
    max_rings_ = std::max(std::min(n, 4096), n / 2);
    const size_t R = (size_t)max_rings_;
    // stamps and counts that only ever grow must start at zero
    const bool fresh = !(mark_.p && mark_.cap >= N * i4);
    MU_TRY(mark_.ensure(N * i4)); MU_TRY(info_.ensure(N * i4)); MU_TRY(extra_n_.ensure(N * i4));
    MU_TRY(list_[0].ensure(N * i4)); MU_TRY(list_[1].ensure(N * i4)); MU_TRY(at_.ensure(N * i4));
    MU_TRY(ring_deg_.ensure(2 * R * i4)); MU_TRY(ring_ref_.ensure(2 * R * kMaxDeg * i4));
    MU_TRY(extra_.ensure(N * kMaxExtra * i4));
    MU_TRY(sizes_.ensure(N * 4)); MU_TRY(images_.ensure(N * 2)); MU_TRY(ghost_off_.ensure((N + 1) * i4));
    MU_TRY(sums_.ensure((size_t)blocks(n, kWindow) * sizeof(int4)));
    MU_TRY(count_.ensure(sizeof(MeshUpdateCount)));
    MU_TRY(flags_.ensure((size_t)n_inst * i4));
    MU_TRY(host_.ensure(sizeof(MeshUpdateCount) + (size_t)n_inst * i4));
    if (fresh || stamp_ > (1 << 28)) {
        MU_TRY(cudaMemsetAsync(mark_.p, 0, mark_.cap, st));
        MU_TRY(cudaMemsetAsync(info_.p, 0, info_.cap, st));
        MU_TRY(cudaMemsetAsync(extra_n_.p, 0, extra_n_.cap, st));
        stamp_ = 0;
    }
    return cudaSuccess;
}

MeshUpdate MeshUpdater::params(const MeshArrays &a) const
{
    MeshUpdate m{};
    m.n = a.n;
    m.n_inst = a.n_inst;
    m.inst = a.inst;
    m.cell_inst = a.cell_inst;
    m.x = a.x;
    m.y = a.y;
    m.cell_ptr = a.cell_ptr;
    m.slot_nb = a.slot_nb;
    m.ghost_src = a.ghost_src;
    m.ghost_img = a.ghost_img;
    m.stamp = stamp_;
    m.mark = mark_.as<int32_t>();
    m.list[0] = list_[0].as<int32_t>();
    m.list[1] = list_[1].as<int32_t>();
    m.ring_info = info_.as<int32_t>();
    m.ring_at = at_.as<int32_t>();
    m.max_rings = max_rings_;
    m.ring_deg = ring_deg_.as<int32_t>();
    m.ring_ref = ring_ref_.as<int32_t>();
    m.extra_n = extra_n_.as<int32_t>();
    m.extra = extra_.as<int32_t>();
    m.count = count_.as<MeshUpdateCount>();
    m.flags = flags_.as<int32_t>();
    m.sizes = sizes_.as<uint32_t>();
    m.images = images_.as<uint16_t>();
    m.ghost_off = ghost_off_.as<int32_t>();
    return m;
}

void MeshUpdater::launch_rounds(const MeshUpdate &m, int first, int last, cudaStream_t st) const
{
    // grids for the cells a step lists (a few per cent), looping beyond
    const int g = std::max(1, std::min(blocks(m.n, 4 * kListBlock), 2048));
    for (int r = first; r < last; r++) {
        k_mesh_recompute<<<g, kListBlock, 0, st>>>(m, r);
        k_mesh_check<<<g, kListBlock, 0, st>>>(m, r);
    }
    const int w = blocks(m.n, kWindow);
    k_mesh_measure<<<w, kWindow, 0, st>>>(m, sums_.as<int4>());
    k_mesh_totals<<<1, kWindow, 0, st>>>(m, sums_.as<int4>(), w);
}

// The rounds launched before the host looks: what nearly every step needs.
constexpr int kFirstRounds = 2;

cudaError_t MeshUpdater::start(const MeshArrays &a, cudaStream_t st)
{
    MU_TRY(reserve(a.n, a.n_inst, st));
    stamp_ += 16;
    static_assert(kMaxRounds + 1 < 16, "one update's stamps");
    const MeshUpdate m = params(a);
    MU_TRY(cudaMemsetAsync(count_.p, 0, sizeof(MeshUpdateCount), st));
    MU_TRY(cudaMemsetAsync(flags_.p, 0, (size_t)a.n_inst * sizeof(int32_t), st));
    k_mesh_verify<<<blocks(a.n, kVerifyBlock), kVerifyBlock, 0, st>>>(m);
    launch_rounds(m, 0, kFirstRounds, st);
    return read_counts(a, st);
}

cudaError_t MeshUpdater::read_counts(const MeshArrays &a, cudaStream_t st)
{
    MU_TRY(cudaMemcpyAsync(host_.p, count_.p, sizeof(MeshUpdateCount), cudaMemcpyDeviceToHost, st));
    MU_TRY(cudaMemcpyAsync(host_.as<MeshUpdateCount>() + 1, flags_.p, (size_t)a.n_inst * sizeof(int32_t),
                           cudaMemcpyDeviceToHost, st));
    return cudaGetLastError();
}

cudaError_t MeshUpdater::settle(const MeshArrays &a, bool &ok, MeshSizes &sizes, cudaStream_t st)
{
    const MeshUpdateCount &c = *host_.as<MeshUpdateCount>();
    int r = kFirstRounds;
    static_assert((kMaxRounds - kFirstRounds) % 2 == 0, "further rounds come in pairs");
    for (; c.listed[r] > 0 && r < kMaxRounds; r += 2) {
        launch_rounds(params(a), r, r + 2, st);
        MU_TRY(read_counts(a, st));
        MU_TRY(cudaStreamSynchronize(st));
    }
    ok = c.listed[r] == 0 && c.slots >= 0 && c.slots <= INT32_MAX / 2;
    const int32_t *f = flags();
    bool flagged = false;
    for (int32_t k = 0; k < a.n_inst; k++) flagged |= f[k] != 0;
    // (what was reported to cells that no round recomputed is dropped)
    if (!ok || flagged) MU_TRY(cudaMemsetAsync(extra_n_.p, 0, extra_n_.cap, st));
    sizes = MeshSizes{c.ghosts, c.tris, c.edges, c.slots};
    return cudaSuccess;
}

const int32_t *MeshUpdater::flags() const { return reinterpret_cast<const int32_t *>(host_.as<MeshUpdateCount>() + 1); }

cudaError_t MeshUpdater::finish(const MeshArrays &a, const MeshOutput &o, cudaStream_t st)
{
    MeshUpdate m = params(a);
    m.out_ptr = o.cell_ptr;
    m.out_nb = o.slot_nb;
    m.tri_off = o.tri_off;
    m.edge_off = o.edge_off;
    m.gx = o.gx;
    m.gy = o.gy;
    m.gsrc = o.ghost_src;
    m.gxf = o.ghost_xf;
    m.gshift = o.ghost_shift;
    m.gimg = o.ghost_img;
    k_mesh_offsets<<<blocks(a.n, kWindow), kWindow, 0, st>>>(m, sums_.as<int4>(), o.cell_order);
    k_mesh_rings<<<blocks(a.n, 256), 256, 0, st>>>(m);
    return cudaGetLastError();
}

}  // namespace rich
