// Kernels of the mesh update (bodies and method: meshupdate.h) and the class
// that holds its device memory.  Compiled without floating-point contraction
// (the predicates' error bounds assume it).
#include "meshupdate_dev.h"

#include <algorithm>

#include "meshupdate.h"

namespace rich {
namespace {

constexpr int kVerifyBlock = 128;  // (as pass_blocks)
constexpr int kListWarps = 4;  // listed cells per block, a warp each
constexpr int kListBlock = 32 * kListWarps;
constexpr int kWindow = kOrderWindow;  // cells per block of the size and ring passes
static_assert(kWindow == 1024, "the scans and the order pass run one window per 1024-thread block");
constexpr unsigned kAll = 0xffffffffu;

// the counters of the next update, cleared by this one's last pass
__device__ __forceinline__ void clear_counters(int32_t *next, int32_t words)
{
    for (int32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < words; k += gridDim.x * blockDim.x) next[k] = 0;
}

// mu::verify<true> with eight lanes per cell, a ring slot each: a thread per
// cell walked its ring through a chain of dependent loads, slot after slot
// (327 us at 1M cells, 24 us at 4,096; now 170 to 330, by how many cells it
// lists, and 9; bound by the latency of its gathers).  Cells of more than eight neighbours
// (3 % of a random mesh) go to the undecided ones.  The warps loop over the
// cells, four at a time, and have the next four's ring slots in flight.
__global__ void __launch_bounds__(kVerifyBlock) k_mesh_verify(MeshUpdate m)
{
    chained(m.n);
    using namespace mu;
    const int lane = threadIdx.x & 31, k = lane & 7, group = lane & 24;
    const unsigned byte = 0xffu << group;
    // a warp lists its cells together: one counter took an atomic for each of
    // the 400,000 cells of a lively step (266 us for this kernel at 1M cells)
    constexpr int kMost = 4 * (8 * 3 + 1);
    __shared__ int32_t listed[kVerifyBlock / 32][kMost];
    __shared__ int32_t listed_n[kVerifyBlock / 32];
    int32_t *cells = listed[threadIdx.x >> 5], *count = &listed_n[threadIdx.x >> 5];
    if (lane == 0) *count = 0;
    const int32_t quads = (m.n + 3) >> 2, stride = gridDim.x * (kVerifyBlock / 32);
    int32_t quad = blockIdx.x * (kVerifyBlock / 32) + (threadIdx.x >> 5);
    auto slots_of = [&](int32_t q, int32_t &i, int32_t &deg, int32_t &id) {
        i = min(4 * q + (group >> 3), m.n - 1);
        const int32_t lo = m.cell_ptr[i];
        deg = m.cell_ptr[i + 1] - lo;
        id = m.slot_nb[lo + (k < deg ? k : 0)];
    };
    int32_t i, deg, id;
    if (quad < quads) slots_of(quad, i, deg, id);
    for (; quad < quads; quad += stride) {
        const bool live = 4 * quad + (group >> 3) < m.n;
        const Frame f = frame_of(m, i);
        const int32_t ref = base_ref(m, id);
        const Point d = point_of(f, ref);
        const bool small = deg <= 8, mine = live && k < deg && small;
        const int last = min(deg, 8) - 1;
        const int32_t cell = i;
        if (quad + stride < quads) slots_of(quad + stride, i, deg, id);
        const int kb = k ? k - 1 : last, ka = kb ? kb - 1 : last;
        Point a, b;
        b.fx = __shfl_sync(kAll, d.fx, group | kb);
        b.fy = __shfl_sync(kAll, d.fy, group | kb);
        b.ref = __shfl_sync(kAll, d.ref, group | kb);
        a.fx = __shfl_sync(kAll, d.fx, group | ka);
        a.fy = __shfl_sync(kAll, d.fy, group | ka);
        a.ref = __shfl_sync(kAll, d.ref, group | ka);
        a.l = a.fx * a.fx + a.fy * a.fy;
        b.l = b.fx * b.fx + b.fy * b.fy;
        const float p = b.fx * d.fy, q = b.fy * d.fx, cbd = p - q;
        const float p3 = a.fx * d.fy, p4 = a.fy * d.fx, p5 = a.fx * b.fy, p6 = a.fy * b.fx;
        const float det = a.l * cbd - b.l * (p3 - p4) + d.l * (p5 - p6);
        const float bound = circle_error(a.l, p, q, b.l, p3, p4, d.l, p5, p6);
        bool bad = -det > bound;
        bool open = !small || !(cbd > cross_error(p, q)) || !(det > bound || bad);
        if (!f.periodic) open = open || ((b.ref & 15) != 4 && (d.ref & 15) != 4);
        open = live && open && (mine || !small);
        bad = bad && mine;
        const bool self = mine && (bad || d.ref != ref || !disk_ok(f, b, d));
        const bool turn = mine && b.fy < 0.0f && d.fy >= 0.0f;
        const unsigned opens = __ballot_sync(kAll, open) & byte, selves = __ballot_sync(kAll, self) & byte;
        const unsigned turns = __ballot_sync(kAll, turn) & byte;
        if (!__any_sync(kAll, live && (opens || selves || __popc(turns) != 1))) continue;
        auto put = [&](int32_t v) {
            if (vol(m.flags + inst_at(m, v)) || vol(m.mark + v) == m.stamp || a_exch(m.mark + v, m.stamp) == m.stamp)
                return;
            cells[atomicAdd(count, 1)] = v;
        };
        if (live && opens) {
            if (k == 0) m.list[1][atomicAdd(&m.count->open, 1)] = cell;
        } else if (live) {
            // (list_bad)
            if (bad) {
                put(b.ref >> 4);
                put(a.ref >> 4);
                put(d.ref >> 4);
                if (f.periodic || (a.ref & 15) == 4) tell_only(m, a.ref >> 4, d.ref);
                if (f.periodic || (d.ref & 15) == 4) tell_only(m, d.ref >> 4, a.ref);
            }
            if (k == 0 && (selves || __popc(turns) != 1)) put(cell);
        }
        __syncwarp();
        const int32_t most = *count;
        int32_t at = 0;
        if (lane == 0 && most > 0) at = atomicAdd(&m.count->listed[0], most);
        at = __shfl_sync(kAll, at, 0);
        for (int32_t t = lane; t < most; t += 32) m.list[0][at + t] = cells[t];
        __syncwarp();
        if (lane == 0) *count = 0;
        __syncwarp();
    }
}

// The cells FP32 left open, a warp each: a lane per ring slot, and for the
// triangles of two images a lane per image that might lie in their circle.
// (A thread per cell spent 127 us on the walls of 4,096 cells; now 18, one
// cell's chain of FP64 and integer predicates.)
// (Two blocks per SM: at the 168 registers that three would leave it spills 96
// bytes, and steps of 50,625 cells take 2 % longer.)
__global__ void __launch_bounds__(kListBlock, 2) k_mesh_verify_open(MeshUpdate m)
{
    chained(m.n);
    using namespace mu;
    const int lane = threadIdx.x & 31;
    const int32_t count = m.count->open;
    for (int32_t c = blockIdx.x * kListWarps + (threadIdx.x >> 5); c < count; c += gridDim.x * kListWarps) {
        const int32_t i = m.list[1][c];
        const Frame f = frame_of(m, i);
        const int32_t lo = m.cell_ptr[i], deg = m.cell_ptr[i + 1] - lo;
        const int32_t *nb = m.slot_nb + lo;
        bool self = false;
        int turns = 0;
        uint32_t imgs = 0;
        if (!f.periodic)
            for (int32_t k = lane; k < deg; k += 32) imgs |= 1u << (base_ref(m, nb[k]) & 15);
        imgs = __reduce_or_sync(kAll, imgs) & ~(1u << 4);
        for (int32_t base = 0; base < deg; base += 32) {
            const int32_t k = base + lane;
            bool pair = false;
            if (k < deg) {
                const int32_t kb = k ? k - 1 : deg - 1, ka = kb ? kb - 1 : deg - 1, ref = base_ref(m, nb[k]);
                const Point a = point_of(f, base_ref(m, nb[ka])), b = point_of(f, base_ref(m, nb[kb]));
                const Point d = point_of(f, ref);
                if (orient_slow(f, b, d) <= 0 || incircle(f, a, b, d) >= 0) {
                    list_bad(m, f.periodic, a.ref, b.ref, d.ref);
                    self = true;
                }
                if (d.ref != ref || !disk_ok_any(f, b, d)) self = true;
                turns += (b.fy < 0.0f && d.fy >= 0.0f) ? 1 : 0;
                pair = !f.periodic && (b.ref & 15) != 4 && (d.ref & 15) != 4;
            }
            for (unsigned pairs = __ballot_sync(kAll, pair); pairs; pairs &= pairs - 1) {
                const int32_t kp = base + __ffs(pairs) - 1;
                const Point b = point_of(f, base_ref(m, nb[kp ? kp - 1 : deg - 1])), d = point_of(f, base_ref(m, nb[kp]));
                for (uint32_t rest = imgs; rest; rest &= rest - 1) {
                    const int img = __ffs((int)rest) - 1;
                    for (int32_t s = lane; s <= deg; s += 32) {
                        const int32_t r = (s == deg ? i : base_ref(m, nb[s]) >> 4) * 16 + img;
                        if (r != b.ref && r != d.ref && incircle(f, b, d, point_of(f, r)) > 0) self = true;
                    }
                }
                __syncwarp();
            }
        }
        turns = __reduce_add_sync(kAll, turns);
        if ((__any_sync(kAll, self) || turns != 1) && lane == 0) list_cell(m, i, 0);
    }
}

// A recomputed star of `deg` neighbours, held one per lane (of `width` lanes
// from lane `first`), into the version that no other cell reads in this round,
// with the cell's sizes.  False when the stars' storage is full.
__device__ __forceinline__ bool commit_star(const MeshUpdate &m, const mu::Frame &f, int32_t round, int32_t ref,
                                            int deg, int first, int width, bool live)
{
    const int lane = threadIdx.x & 31, k = lane - first;
    const int32_t info = m.ring_info[f.i];
    const bool fresh = (info >> 2) < m.stamp;
    int32_t place = 0;
    if (live && k == 0) place = fresh ? atomicAdd(&m.count->overrides, 1) : m.ring_at[f.i];
    place = __shfl_sync(kAll, place, first);
    const bool fits = place < m.max_rings;
    const int32_t ver = fresh ? 0 : (info & 1) ^ 1;
    // owned edges and triangles (mu::ring_sizes)
    const int32_t prev = __shfl_sync(kAll, ref, first + (k ? k - 1 : deg - 1 < 0 ? 0 : deg - 1));
    const bool in = live && k < deg;
    const bool up = (ref & 15) != 4 || (ref >> 4) > f.i, prev_up = (prev & 15) != 4 || (prev >> 4) > f.i;
    const bool edge = (ref & 15) == 4 || f.periodic ? (ref >> 4) > f.i : true;
    const unsigned group = width == 32 ? kAll : ((1u << width) - 1) << first;
    const unsigned ne = __ballot_sync(kAll, in && edge) & group, nt = __ballot_sync(kAll, in && up && prev_up) & group;
    if (in && fits) m.ring_ref[(int64_t)(2 * place + ver) * kMaxDeg + k] = ref;
    if (live && k == 0) {
        if (!fits) {
            mu::a_or(f.flags, MU_SIZE);
        } else {
            if (fresh) m.ring_at[f.i] = place;
            m.ring_deg[2 * place + ver] = deg;
            m.ring_info[f.i] = (m.stamp + round) << 2 | (fresh ? 2 : 0) | ver;
            m.sizes[f.i] = (uint32_t)deg | __popc(ne) << 8 | __popc(nt) << 16;
        }
        m.extra_n[f.i] = 0;
    }
    return fits;
}

// mu::recompute_light for the first round's cells, a lane per candidate and
// sixteen lanes per cell: the wrapping finds each next neighbour by a
// tournament.  (A thread per cell took as long at 4,096 cells, 48 us, as at
// 262,144: one cell's chain of steps.  Now 11 us, and 32 to 50 with 7,500 to
// 39,000 cells listed of 262,144, bound by instruction issue.)
__global__ void __launch_bounds__(kListBlock) k_mesh_recompute_light(MeshUpdate m)
{
    chained(m.n);
    using namespace mu;
    static_assert(kLight == 16, "a half warp per cell");
    const int lane = threadIdx.x & 31, c = lane & 15, first = lane & 16;
    const unsigned half = 0xffffu << first;
    const int32_t count = m.count->listed[0];
    for (int32_t k0 = (blockIdx.x * kListWarps + (threadIdx.x >> 5)) * 2; k0 < count; k0 += gridDim.x * kListWarps * 2) {
        const int32_t kk = k0 + (first >> 4);
        const bool live = kk < count;
        const int32_t i = m.list[0][live ? kk : k0];
        const Frame f = frame_of(m, i);
        const Ring own = ring_of(m, i, 0);
        const int32_t ne = m.extra_n[i], n = own.deg + ne;
        bool ok = live && n <= kLight && ne <= kMaxExtra;
        int32_t r = i * 16 + 4;
        if (c < own.deg) r = own[c];
        else if (c < n && ne <= kMaxExtra) r = m.extra[(int64_t)i * kMaxExtra + (c - own.deg)];
        bool mine = c < n;
        // a cell at a wall, or an image of itself, goes to the full recomputation
        if (mine && ((!f.periodic && (r & 15) != 4) || (r >> 4) == i)) ok = false;
        ok = (__ballot_sync(kAll, ok) & half) == half;
        for (int t = 0; t < 15; t++) {
            const int32_t s = __shfl_sync(kAll, r, first + t);
            if (t < c && (s >> 4) == (r >> 4)) mine = false;
        }
        const Point d = point_of(f, r);
        // (the nearest in FP32 is a neighbour unless another candidate lies
        // within a thousandth of its distance of it; the wrapping then does
        // not close)
        float lmin = mine ? d.l : __int_as_float(0x7f800000);
        int near = c;
        for (int o = 8; o > 0; o >>= 1) {
            const float l2 = __shfl_xor_sync(kAll, lmin, o);
            const int n2 = __shfl_xor_sync(kAll, near, o);
            if (l2 < lmin || (l2 == lmin && n2 < near)) {
                lmin = l2;
                near = n2;
            }
        }
        int deg = 0, last = near, turns = 0, kept = 0;
        bool open = ok;
        while (__any_sync(kAll, open)) {
            if (c == deg) kept = last;
            Point a;
            a.fx = __shfl_sync(kAll, d.fx, first + last);
            a.fy = __shfl_sync(kAll, d.fy, first + last);
            a.l = a.fx * a.fx + a.fy * a.fy;
            const float p = a.fx * d.fy, q = a.fy * d.fx, cr = p - q, cb = cross_error(p, q);
            const bool cand = mine && c != last;
            bool unsure = cand && !(cr > cb) && !(-cr > cb);
            int best = cand && cr > cb ? c : -1;
            for (int o = 8; o > 0; o >>= 1) {
                const int other = __shfl_xor_sync(kAll, best, o);
                const int sb = first + (best < 0 ? 0 : best), so = first + (other < 0 ? 0 : other);
                Point b, e;
                b.fx = __shfl_sync(kAll, d.fx, sb);
                b.fy = __shfl_sync(kAll, d.fy, sb);
                e.fx = __shfl_sync(kAll, d.fx, so);
                e.fy = __shfl_sync(kAll, d.fy, so);
                if (other < 0 || other == best) continue;
                if (best < 0) {
                    best = other;
                    continue;
                }
                b.l = b.fx * b.fx + b.fy * b.fy;
                e.l = e.fx * e.fx + e.fy * e.fy;
                const float p1 = b.fx * e.fy, p2 = b.fy * e.fx, p3 = a.fx * e.fy, p4 = a.fy * e.fx, p5 = a.fx * b.fy,
                            p6 = a.fy * b.fx;
                const float det = a.l * (p1 - p2) - b.l * (p3 - p4) + e.l * (p5 - p6);
                const float bound = circle_error(a.l, p1, p2, b.l, p3, p4, e.l, p5, p6);
                if (-det > bound) best = other;
                else if (!(det > bound)) unsure = true;
            }
            const int nb = first + (best < 0 ? 0 : best);
            Point b;
            b.fx = __shfl_sync(kAll, d.fx, nb);
            b.fy = __shfl_sync(kAll, d.fy, nb);
            b.l = b.fx * b.fx + b.fy * b.fy;
            const bool fail = unsure || best < 0 || !disk_ok(f, a, b);
            const bool failed = (__ballot_sync(kAll, fail) & half) != 0;
            if (open) {
                deg++;
                turns += (a.fy < 0.0f && b.fy >= 0.0f) ? 1 : 0;
                last = best;
                if (failed || (deg == kLight && last != near)) ok = open = false;
                else if (last == near) open = false;
            }
        }
        ok = ok && deg >= 3 && turns == 1;
        const int32_t ref = __shfl_sync(kAll, d.ref, first + kept);
        commit_star(m, f, 0, ref, deg, first, 16, ok);
        if (live && !ok && c == 0) m.heavy[atomicAdd(&m.count->heavy, 1)] = i;
    }
}

// One warp's working set for one cell.
struct StarWork {
    int32_t src[kMaxSources];
    int32_t ref[kMaxCand];
    float fx[kMaxCand], fy[kMaxCand];
    int32_t out[kMaxDeg];
};

// mu::recompute with a warp per cell: the lanes read the neighbours' rings,
// drop repeated sources, take a candidate or two each, and find the next
// neighbour of the gift wrapping by a tournament of in-circle tests.  A step
// lists a few hundred to a few per cent of the cells, so the pass is bound by
// one cell's chain of dependent loads and tests: a thread per cell took 545 us
// at 1M cells and 540 us for the wall cells of 4,096; now 13 us for 200 cells
// at walls.
__device__ void warp_recompute(const MeshUpdate &m, int32_t i, int32_t round, StarWork &w)
{
    using namespace mu;
    const int lane = threadIdx.x & 31;
    const Frame f = frame_of(m, i);
    const Ring own = ring_of(m, i, round);
    const int32_t told = m.extra_n[i], ne = told < kMaxExtra ? told : kMaxExtra;
    __syncwarp();
    if (lane == 0) m.extra_n[i] = 0;
    if (own.deg + ne > 32) {
        if (lane == 0) a_or(f.flags, MU_SIZE);
        return;
    }
    // this lane's neighbour (or vertex told of), and its ring
    const int first = own.deg + ne;
    int32_t r = i * 16 + 4;
    if (lane < own.deg) r = own[lane];
    else if (lane < first) r = m.extra[(int64_t)i * kMaxExtra + (lane - own.deg)];
    uint32_t imgs = 1u << (r & 15);
    const bool far_own = (r >> 4) == i;  // an image of the cell itself (or no neighbour)
    const Ring g = ring_of(m, r >> 4, round);
    const int mine = far_own ? 0 : g.deg;
    int at = mine;
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(kAll, at, o);
        if (lane >= o) at += u;
    }
    const int total = first + __shfl_sync(kAll, at, 31);
    at += first - mine;
    if (total > kMaxSources) {
        if (lane == 0) a_or(f.flags, MU_SIZE);
        return;
    }
    if (lane < first) w.src[lane] = r >> 4;
    for (int j = 0; j < mine; j++) {
        const int32_t q = g[j];
        imgs |= 1u << (q & 15);
        w.src[at + j] = q >> 4;
    }
    imgs = __reduce_or_sync(kAll, imgs);
    __syncwarp();
    // distinct sources, the cell left out, to the front
    int ns = 0;
    for (int base = 0; base < total; base += 32) {
        const int k = base + lane;
        const int32_t s = k < total ? w.src[k] : i;
        bool keep = s != i;
        // (entries before this batch are the ones kept so far)
        for (int q = 0; q < ns; q++) keep = keep && w.src[q] != s;
        const unsigned same = __match_any_sync(kAll, s);
        keep = keep && (same & ((1u << lane) - 1)) == 0;
        const unsigned kept = __ballot_sync(kAll, keep);
        __syncwarp();
        // (place ns + rank is at most k: an entry already read)
        if (keep) w.src[ns + __popc(kept & ((1u << lane) - 1))] = s;
        __syncwarp();
        ns += __popc(kept);
    }
    // the candidates: every source, and across walls every image that these
    // rings meet, of the cell too
    const bool walls = !f.periodic && (imgs & ~(1u << 4)) != 0;
    const int per = walls ? ns + 1 : ns, sets = walls ? __popc(imgs | 1u << 4) : 1;
    const int nc = per * sets;
    if (nc > kMaxCand || nc < 3) {
        if (lane == 0) a_or(f.flags, MU_SIZE);
        return;
    }
    // (the cell itself, image 4 of the walls' sets, is no candidate)
    unsigned long long dmin = ~0ull;
    int near = -1;
    for (int c = lane; c < nc; c += 32) {
        int img = 4, k = c;
        if (walls) {
            uint32_t rest = imgs | 1u << 4;
            for (; k >= per; k -= per) rest &= rest - 1;
            img = __ffs((int)rest) - 1;
        }
        const int32_t src = k < ns ? w.src[k] : i;
        if (src == i && img == 4) {
            w.ref[c] = -1;
            continue;
        }
        const Point p = point_of(f, src * 16 + img);
        w.ref[c] = p.ref;
        w.fx[c] = p.fx;
        w.fy[c] = p.fy;
        const double dx = p.x - f.xi, dy = p.y - f.yi;
        const unsigned long long d2 = (unsigned long long)__double_as_longlong(dx * dx + dy * dy);
        if (d2 < dmin) {
            dmin = d2;
            near = c;
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long d = __shfl_xor_sync(kAll, dmin, o);
        const int n2 = __shfl_xor_sync(kAll, near, o);
        if (d < dmin || (d == dmin && n2 > near)) {
            dmin = d;
            near = n2;
        }
    }
    __syncwarp();
    auto at_of = [&](int c) {
        Point p;
        p.ref = w.ref[c];
        p.fx = w.fx[c];
        p.fy = w.fy[c];
        p.l = p.fx * p.fx + p.fy * p.fy;
        return p;
    };
    // whether candidate d is inside the circle of (cell, a, b)
    auto inside = [&](const Point &a, int b, int d) {
        const Point pb = at_of(b), pd = at_of(d);
        const float p1 = pb.fx * pd.fy, p2 = pb.fy * pd.fx, p3 = a.fx * pd.fy, p4 = a.fy * pd.fx, p5 = a.fx * pb.fy,
                    p6 = a.fy * pb.fx;
        const float det = a.l * (p1 - p2) - pb.l * (p3 - p4) + pd.l * (p5 - p6);
        const float bound = circle_error(a.l, p1, p2, pb.l, p3, p4, pd.l, p5, p6);
        if (det > bound) return false;
        if (-det > bound) return true;
        return circle_slow(f, a.ref, pb.ref, pd.ref) > 0;
    };
    int deg = 0, last = near, turns = 0;
    bool bad = false;
    do {
        if (deg == kMaxDeg) {
            bad = true;
            break;
        }
        const Point a = at_of(last);
        if (lane == 0) w.out[deg] = a.ref;
        deg++;
        int best = -1;
        for (int c = lane; c < nc; c += 32) {
            if (c == last || w.ref[c] < 0) continue;
            const float p = a.fx * w.fy[c], q = a.fy * w.fx[c], cr = p - q;
            const float cb = cross_error(p, q);
            bool left = cr > cb;
            if (!left && !(-cr > cb)) left = orient_slow(f, a.ref, w.ref[c]) > 0;
            if (left && (best < 0 || inside(a, best, c))) best = c;
        }
        __syncwarp();
        for (int o = 16; o > 0; o >>= 1) {
            const int other = __shfl_xor_sync(kAll, best, o);
            if (other >= 0 && other != best && (best < 0 || inside(a, best, other))) best = other;
            __syncwarp();
        }
        if (best < 0) {
            bad = true;
            break;
        }
        const Point b = at_of(best);
        if (lane == 0 && !disk_ok_any(f, a, b)) a_or(f.flags, MU_FAR);
        turns += (a.fy < 0.0f && b.fy >= 0.0f) ? 1 : 0;
        last = best;
    } while (last != near);
    __syncwarp();
    if (bad || deg < 3 || turns != 1) {
        if (lane == 0) a_or(f.flags, MU_STAR);
        return;
    }
    commit_star(m, f, round, lane < deg ? w.out[lane] : 0, deg, 0, 32, true);
}

// (Two blocks per SM, 209 registers: at the 168 that three would leave it spills
// 44 bytes, 18.7 us for the walls of 4,096 cells instead of 17.1, and 698
// instead of 713 for a batch of 4.5M cells, most beside walls.  Absolute
// positions kept in shared memory gain 80 us there, but the larger carve-out
// costs every small step 11 us.)
__global__ void __launch_bounds__(kListBlock, 2) k_mesh_recompute(MeshUpdate m, int32_t round)
{
    chained(m.n);
    __shared__ StarWork work[kListWarps];
    const int32_t count = round ? m.count->listed[round] : m.count->heavy;
    const int32_t *list = round ? m.list[round & 1] : m.heavy;
    for (int32_t k = blockIdx.x * kListWarps + (threadIdx.x >> 5); k < count; k += gridDim.x * kListWarps) {
        warp_recompute(m, list[k], round, work[threadIdx.x >> 5]);
        __syncwarp();
    }
}

// eight lanes per cell, one per triangle and per dropped neighbour
__global__ void __launch_bounds__(kListBlock) k_mesh_check(MeshUpdate m, int32_t round)
{
    chained(m.n);
    const int t = threadIdx.x & 7;
    const int32_t count = m.count->listed[round], cells = kListBlock / 8;
    for (int32_t k = blockIdx.x * cells + (threadIdx.x >> 3); k < count; k += gridDim.x * cells) {
        const int32_t i = m.list[round & 1][k];
        if (!mu::recomputed(m, i, round)) continue;
        const bool periodic = m.inst[mu::inst_at(m, i)].boundary == 1;
        const mu::Ring g = mu::ring_of(m, i, -1), old = mu::ring_of(m, i, round);
        for (int32_t q = t; q < g.deg; q += 8) mu::check_triangle(m, periodic, g, i, round, q);
        for (int32_t q = t; q < old.deg; q += 8) mu::check_dropped(m, periodic, g, old, i, round, q);
    }
}

// The simulations of cells still listed for `round`: theirs are left to the
// host, and the others' meshes can be written.
__global__ void k_mesh_give_up(MeshUpdate m, int32_t round)
{
    const int32_t count = m.count->listed[round];
    for (int32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < count; k += gridDim.x * blockDim.x)
        mu::a_or(m.flags + mu::inst_at(m, m.list[round & 1][k]), MU_ROUNDS);
}

__device__ __forceinline__ int4 plus(int4 a, int4 b) { return make_int4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }

__device__ __forceinline__ int4 warp_total(int4 v)
{
    v.x = __reduce_add_sync(kAll, v.x);
    v.y = __reduce_add_sync(kAll, v.y);
    v.z = __reduce_add_sync(kAll, v.z);
    v.w = __reduce_add_sync(kAll, v.w);
    return v;
}

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

// Sizes per cell and their sums per window.  A mesh's sizes are kept: the
// recomputations set those of the rings they change, so that only the images
// inside the ghost band are counted again (whole: every ring is measured, for
// a mesh that the host built).
__global__ void __launch_bounds__(kWindow) k_mesh_measure(MeshUpdate m, int4 *window_sums, int32_t whole)
{
    chained(m.n);
    __shared__ int4 part[32];
    const int32_t i = blockIdx.x * kWindow + threadIdx.x;
    int4 v = make_int4(0, 0, 0, 0);
    if (i < m.n) v = sizes_of(whole ? mu::measure(m, i) : m.sizes[i] = mu::count_images(m, i, m.sizes[i]));
    v = warp_total(v);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        v = warp_total(part[threadIdx.x]);
        if (threadIdx.x == 0) window_sums[blockIdx.x] = v;
    }
}

// offsets per cell, the ghosts, and the processing order: within each window
// cells by decreasing ring degree, stable (degree_order in mesh.cpp)
// Every block adds up the windows before its own, and all of them: the mesh
// can be written when no cell is listed for round `last` and it fits its
// arrays.
__global__ void __launch_bounds__(kWindow) k_mesh_offsets(MeshUpdate m, int4 *window_sums, int32_t last)
{
    chained(m.n);
    __shared__ int4 totals[2];
    {
        __shared__ int4 part[2][32];
        const int w = threadIdx.x >> 5;
        int4 before = make_int4(0, 0, 0, 0), all = before;
        for (int32_t k = threadIdx.x; k < (int32_t)gridDim.x; k += kWindow) {
            const int4 v = window_sums[k];
            all = plus(all, v);
            if (k < (int32_t)blockIdx.x) before = plus(before, v);
        }
        all = warp_total(all);
        before = warp_total(before);
        if ((threadIdx.x & 31) == 0) {
            part[0][w] = before;
            part[1][w] = all;
        }
        __syncthreads();
        if (w < 2) {
            const int4 t = warp_total(part[w][threadIdx.x & 31]);
            if ((threadIdx.x & 31) == 0) totals[w] = t;
        }
        __syncthreads();
        const int4 t = totals[1];
        const bool fits = t.x >= 0 && t.x <= m.max_slots && t.y <= m.max_edges && t.z <= m.max_tris && t.w <= m.max_ghosts;
        const bool ready = fits && m.count->listed[last] == 0 && !(m.n_inst == 1 && m.flags[0]);
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            m.count->slots = t.x;
            m.count->edges = t.y;
            m.count->tris = t.z;
            m.count->ghosts = t.w;
            m.count->ready = ready ? 1 : 0;
        }
        if (!ready) return;
    }
    __shared__ int4 ws[32];
    __shared__ int32_t of_degree[65];
    __shared__ int32_t hist[32][65];  // cells of each degree in each warp, then their first places
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int32_t i = blockIdx.x * kWindow + threadIdx.x;
    const int4 own = i < m.n ? sizes_of(m.sizes[i]) : make_int4(0, 0, 0, 0);
    const int4 inc = block_sum(own, ws), base = totals[0];
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
        of_degree[threadIdx.x] = run;  // cells of this degree in the window
    }
    __syncthreads();
    if (wid == 0) {
        // cells of larger degrees: sums from 64 down, two and then 64's own
        int lo = of_degree[lane], hi = of_degree[32 + lane];
        const int top = of_degree[64];
        for (int o = 1; o < 32; o <<= 1) {
            const int a = __shfl_down_sync(kAll, lo, o), b = __shfl_down_sync(kAll, hi, o);
            if (lane + o < 32) {
                lo += a;
                hi += b;
            }
        }
        const int all_hi = __shfl_sync(kAll, hi, 0);
        __syncwarp();
        // (exclusive: minus the degree's own)
        of_degree[lane] = lo - of_degree[lane] + all_hi + top;
        of_degree[32 + lane] = hi - of_degree[32 + lane] + top;
        if (lane == 0) of_degree[64] = 0;
    }
    __syncthreads();
    if (deg >= 0) {
        const int place = of_degree[deg] + hist[wid][deg] + before;
        m.cell_order[blockIdx.x * kWindow + place] = i;
    }
}

// mu::place_ring with eight lanes per cell, and the masks of each ring's
// owned edges and triangles (cells of up to 32 neighbours), from which
// k_mesh_lists takes every edge's and triangle's number.  A ring that no round
// changed and that meets no image keeps its ids and their order.
__global__ void __launch_bounds__(128) k_mesh_rings(MeshUpdate m)
{
    chained(m.n);
    if (!m.count->ready) return;
    using namespace mu;
    const int lane = threadIdx.x & 31, k = lane & 7, first = lane & 24;
    const int32_t quads = (m.n + 3) >> 2, stride = gridDim.x * (blockDim.x >> 5);
    for (int32_t quad = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); quad < quads; quad += stride) {
        const int32_t t = 4 * quad + (first >> 3);
        const bool live = t < m.n;
        const int32_t i = live ? t : m.n - 1;
        const Ring g = ring_of(m, i, -1);
        const bool periodic = m.inst[inst_at(m, i)].boundary == 1;
        int32_t *dst = m.out_nb + m.out_ptr[i];
        if (__all_sync(kAll, g.deg <= 8)) {
            const bool in = live && k < g.deg;
            const int32_t q = k < g.deg ? k : 0;
            const bool plain = g.base && g.p[q] < m.n;
            int32_t id = plain ? g.p[q] : 0;
            int at = 0;
            if (!__all_sync(kAll, plain)) {
                if (!plain) id = point_id(m, i, g[q]);
                int32_t best = id;
                at = q;
                for (int o = 4; o > 0; o >>= 1) {
                    const int32_t b2 = __shfl_xor_sync(kAll, best, o), a2 = __shfl_xor_sync(kAll, at, o);
                    if (b2 < best || (b2 == best && a2 < at)) {
                        best = b2;
                        at = a2;
                    }
                }
            }
            const int pos = q >= at ? q - at : q - at + g.deg;
            const int32_t next = __shfl_sync(kAll, id, first + (q + 1 < g.deg ? q + 1 : 0));
            // (an image owns nothing; whether the cell owns a periodic edge to
            // one follows from the source: images of the cell itself have no
            // place in an updated mesh)
            const bool edge = id < m.n || !periodic ? id > i : (g[q] >> 4) > i;
            uint32_t own = in ? (edge ? 1u << pos : 0u) | (id > i && next > i ? 256u << pos : 0u) : 0u;
            for (int o = 4; o > 0; o >>= 1) own |= __shfl_xor_sync(kAll, own, o);
            if (in) dst[pos] = id;
            if (live && k == 0) {
                m.edge_mask[i] = own & 255u;
                m.tri_mask[i] = own >> 8;
            }
            continue;
        }
        // some ring of the warp has more than eight members
        int32_t best = INT32_MAX, at = 0;
        for (int32_t q = k; q < g.deg; q += 8) {
            const int32_t id = point_id(m, i, g[q]);
            if (id < best) {
                best = id;
                at = q;
            }
        }
        for (int o = 4; o > 0; o >>= 1) {
            const int32_t b2 = __shfl_xor_sync(kAll, best, o), a2 = __shfl_xor_sync(kAll, at, o);
            if (b2 < best || (b2 == best && a2 < at)) {
                best = b2;
                at = a2;
            }
        }
        uint32_t edges = 0, tris = 0;
        for (int32_t q = k; q < g.deg; q += 8) {
            const int32_t pos = q >= at ? q - at : q - at + g.deg, r = g[q];
            const int32_t id = point_id(m, i, r), next = point_id(m, i, g[q + 1 < g.deg ? q + 1 : 0]);
            if (live) dst[pos] = id;
            if (pos < 32) {
                if (id < m.n || !periodic ? id > i : (r >> 4) > i) edges |= 1u << pos;
                if (id > i && next > i) tris |= 1u << pos;
            }
        }
        for (int o = 4; o > 0; o >>= 1) {
            edges |= __shfl_xor_sync(kAll, edges, o);
            tris |= __shfl_xor_sync(kAll, tris, o);
        }
        if (live && k == 0) {
            m.edge_mask[i] = edges;
            m.tri_mask[i] = tris;
        }
    }
}

// owner of the edge between real cell i and point j (1: i, 0: the other
// side, -1: inconsistent), the host builder's rule
__device__ __forceinline__ int edge_owner(const MeshLists &l, bool periodic, int32_t i, int32_t j)
{
    if (j < l.n) return j > i ? 1 : (j < i ? 0 : -1);
    if (!periodic) return 1;
    const int32_t src = l.ghost_src[j - l.n];
    if (src != i) return src > i ? 1 : 0;
    const int32_t sh = l.ghost_shift[j - l.n];
    const int32_t sx = sh % 3 - 1, sy = sh / 3 - 1;
    return (sy < 0 || (sy == 0 && sx < 0)) ? 0 : 1;
}

// The lists of four cells (eight lanes each) of any degree, in a mesh of the
// update or of the host: k_mesh_lists for the cells that its own code, for
// rings of up to eight with masks, does not take.
__device__ __noinline__ bool lists_of_any(const MeshLists &l, int32_t i, bool live, bool periodic)
{
    const int lane = threadIdx.x & 31, k = lane & 7, first = lane & 24;
    const unsigned byte = 0xffu << first, below = ((1u << k) - 1) << first;
    const int32_t lo = l.cell_ptr[i], deg = l.cell_ptr[i + 1] - lo;
    const int32_t *nb = l.slot_nb + lo;
    int32_t t = l.tri_off[i], e = l.edge_off[i];
    const int32_t t_end = l.tri_off[i + 1], e_end = l.edge_off[i + 1];
    bool bad = false;
    int owner = -1;
    // the loops run as long as any cell of the warp has slots
    const int32_t steps = __reduce_max_sync(kAll, (deg + 7) >> 3);
    for (int32_t s = 0; s < steps; s++) {
        const int32_t q = 8 * s + k;
        const bool in = live && q < deg;
        const int32_t a = nb[in ? q : 0], b = nb[in && q + 1 < deg ? q + 1 : 0];
        const bool own_tri = in && i < a && i < b;
        const unsigned tris = __ballot_sync(kAll, own_tri) & byte;
        if (own_tri) {
            const int32_t num = t + __popc(tris & below);
            if (num < t_end) {
                l.tri[3 * num] = i;
                l.tri[3 * num + 1] = a;
                l.tri[3 * num + 2] = b;
                l.slot_tri[lo + q] = num;
            } else {
                bad = true;
            }
        }
        t += __popc(tris);
        if (in) {
            owner = edge_owner(l, periodic, i, a);
            if (owner < 0) bad = true;
        }
        if (in && a < i) {
            // this cell in the ring of a: edges and triangles of a before it
            const int32_t prev = nb[q ? q - 1 : deg - 1];
            const int32_t alo = l.cell_ptr[a], adeg = l.cell_ptr[a + 1] - alo;
            const int32_t *an = l.slot_nb + alo;
            int32_t ne = l.edge_off[a], nt = l.tri_off[a];
            bool found = false;
            int32_t j0 = 0;
            if (l.edge_mask && adeg <= 32) {
                while (j0 < adeg && an[j0] != i) j0++;
                if (j0 < adeg) {
                    const uint32_t passed = (1u << j0) - 1;
                    ne += __popc(l.edge_mask[a] & passed);
                    nt += __popc(l.tri_mask[a] & passed);
                }
            }
            int32_t x = j0 < adeg ? an[j0] : -1, before = an[j0 ? j0 - 1 : adeg - 1];
            for (int32_t j = j0; j < adeg; j++) {
                const int32_t y = an[j + 1 < adeg ? j + 1 : 0];
                if (x == i) {
                    // (a; before, i) is this slot's triangle, (a; i, y) the last slot's
                    l.slot_edge[lo + q] = 2 * ne + 1;
                    if (a < b) {
                        if (before != b) bad = true;
                        l.slot_tri[lo + q] = j ? nt - 1 : l.tri_off[a + 1] - 1;
                    }
                    if (a < prev) {
                        if (y != prev) bad = true;
                        l.slot_tri[lo + (q ? q - 1 : deg - 1)] = nt;
                    }
                    found = true;
                    break;
                }
                ne += edge_owner(l, periodic, a, x) > 0 ? 1 : 0;
                nt += a < x && a < y ? 1 : 0;
                before = x;
                x = y;
            }
            if (!found) bad = true;
        } else if (in && a >= l.n && owner == 0) {
            // a periodic edge that the source of a owns: from its ring this
            // cell is seen at the opposite shift
            const int32_t src = l.ghost_src[a - l.n], sh = l.ghost_shift[a - l.n];
            const int32_t want = (1 - (sh % 3 - 1)) + 3 * (1 - (sh / 3 - 1));
            const int32_t alo = l.cell_ptr[src], adeg = l.cell_ptr[src + 1] - alo;
            int32_t ne = l.edge_off[src];
            bool found = false;
            for (int32_t j = 0; j < adeg; j++) {
                const int32_t x = l.slot_nb[alo + j];
                if (x >= l.n && l.ghost_src[x - l.n] == i && l.ghost_shift[x - l.n] == want && alo + j != lo + q) {
                    l.slot_edge[lo + q] = 2 * ne + 1;
                    found = true;
                    break;
                }
                ne += edge_owner(l, periodic, src, x) > 0 ? 1 : 0;
            }
            if (!found) bad = true;
        }
    }
    if (live && t != t_end) bad = true;
    // the owned edges, whose triangles are now all numbered
    __syncwarp();
    for (int32_t s = 0; s < steps; s++) {
        const int32_t q = 8 * s + k;
        const bool in = live && q < deg;
        const int32_t a = nb[in ? q : 0];
        const bool own = in && edge_owner(l, periodic, i, a) > 0;
        const unsigned edges = __ballot_sync(kAll, own) & byte;
        if (own) {
            const int32_t num = e + __popc(edges & below);
            if (num < e_end) {
                l.edge_l[num] = i;
                l.edge_r[num] = a;
                l.edge_ta[num] = *(volatile const int32_t *)(l.slot_tri + lo + (q ? q - 1 : deg - 1));
                l.edge_tb[num] = *(volatile const int32_t *)(l.slot_tri + lo + q);
                l.slot_edge[lo + q] = 2 * num;
            } else {
                bad = true;
            }
        }
        e += __popc(edges);
    }
    if (live && e != e_end) bad = true;
    return bad;
}

// The update's counters to the host, by the block that ends last (a copy after
// the kernel is 2 to 3 us more of a small step's chain).
__device__ __forceinline__ void report_counters(const MeshLists &l)
{
    if (!l.report) return;
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(l.done, 1) == (int32_t)gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int32_t k = threadIdx.x; k < l.words; k += blockDim.x) l.report[k] = __ldcg(l.counters + k);
    if (threadIdx.x == 0) *l.done = 0;
}

// The triangle and edge lists from the rings, eight lanes per cell, a ring
// slot each.  A slot whose neighbour is a smaller real cell finds this cell in
// that one's ring: the edges and triangles that the neighbour owns before it
// (from the masks of k_mesh_rings, or counted on the way in a mesh that the
// host built) number the edge and both triangles beside it, so every slot is
// written once, by its own cell, and needs no clearing and no later check.
// (Three kernels before: triangles and edges with a walk per triangle and
// per edge, and a check of both, 153 us at 1M cells with every block resident;
// now 126 so, and 205 in the fewer blocks that run beside the FP64 stages.)
__global__ void __launch_bounds__(128, 8) k_mesh_lists(MeshLists l)
{
    chained(l.n);
    if (l.next) clear_counters(l.next, l.next_words);
    if (l.ready && !*l.ready) {
        report_counters(l);
        return;
    }
    const int lane = threadIdx.x & 31, k = lane & 7, first = lane & 24;
    const int32_t quads = (l.n + 3) >> 2, stride = gridDim.x * (blockDim.x >> 5);
    // (a cell's lists are its simulation's: another's are good all the same)
    auto report_bad = [&](int32_t i) {
        *l.bad = 1;
        if (l.flags) atomicOr(l.flags + (l.cell_inst ? l.cell_inst[i] : 0), (int32_t)MU_LISTS);
    };
    for (int32_t quad = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); quad < quads; quad += stride) {
        bool bad = false;
        const int32_t cell = 4 * quad + (first >> 3);
        const bool live = cell < l.n;
        const int32_t i = live ? cell : l.n - 1;
        const bool periodic = l.cell_inst ? l.inst[l.cell_inst[i]].boundary == 1 : l.periodic != 0;
        const int32_t lo = l.cell_ptr[i], deg = l.cell_ptr[i + 1] - lo;
        if (!__all_sync(kAll, l.edge_mask && deg <= 8)) {
            if (lists_of_any(l, i, live, periodic)) report_bad(i);
            continue;
        }
        const int q = k < deg ? k : 0;
        const int32_t t0 = l.tri_off[i], e0 = l.edge_off[i];
        const int32_t own_edges = (int32_t)l.edge_mask[i], own_tris = (int32_t)l.tri_mask[i];
        // (a mesh left to the host may not agree with its counts)
        const bool counted = __popc(own_tris) == l.tri_off[i + 1] - t0 && __popc(own_edges) == l.edge_off[i + 1] - e0;
        const bool in = live && counted && k < deg;
        bad |= !counted;
        const int32_t a = l.slot_nb[lo + q];
        const int32_t b = __shfl_sync(kAll, a, first + (q + 1 < deg ? q + 1 : 0));
        const int32_t prev = __shfl_sync(kAll, a, first + (q ? q - 1 : deg - 1));
        const bool own_tri = in && (own_tris >> q & 1), own_edge = in && (own_edges >> q & 1);
        // this slot's triangle and the one before it, where known here
        int32_t tri = own_tri ? t0 + __popc(own_tris & ((1 << q) - 1)) : -1, tri_before = -1;
        if (own_tri) {
            l.tri[3 * tri] = i;
            l.tri[3 * tri + 1] = a;
            l.tri[3 * tri + 2] = b;
        }
        if (in && a < i) {
            const int32_t alo = l.cell_ptr[a], adeg = l.cell_ptr[a + 1] - alo;
            const uint32_t em = l.edge_mask[a], tm = l.tri_mask[a];
            const int32_t te = l.tri_off[a + 1], ta = l.tri_off[a], ea = l.edge_off[a];
            const int32_t *an = l.slot_nb + alo;
            // (eight loads at once: a loop would wait for each)
            int32_t ring[8];
#pragma unroll
            for (int c = 0; c < 8; c++) ring[c] = c < adeg ? an[c] : -1;
            int32_t at = adeg;
#pragma unroll
            for (int c = 7; c >= 0; c--) at = ring[c] == i ? c : at;
            if (at == adeg)
                for (at = 8; at < adeg && an[at] != i; at++) {}
            if (at >= adeg || adeg > 32) {
                bad = true;
            } else {
                const uint32_t passed = (1u << at) - 1;
                const int32_t ne = ea + __popc(em & passed), nt = ta + __popc(tm & passed);
                l.slot_edge[lo + q] = 2 * ne + 1;
                // (a; b, i) is this slot's triangle, (a; i, prev) the one before
                if (a < b) {
                    bad |= an[at ? at - 1 : adeg - 1] != b;
                    tri = at ? nt - 1 : te - 1;
                }
                if (a < prev) {
                    bad |= an[at + 1 < adeg ? at + 1 : 0] != prev;
                    tri_before = nt;
                }
            }
        } else if (in && !own_edge) {
            // a periodic edge that the source of a owns: from its ring this
            // cell is seen at the opposite shift
            bool found = false;
            if (a >= l.n) {
                const int32_t src = l.ghost_src[a - l.n], sh = l.ghost_shift[a - l.n];
                const int32_t want = (1 - (sh % 3 - 1)) + 3 * (1 - (sh / 3 - 1));
                const int32_t alo = l.cell_ptr[src], adeg = l.cell_ptr[src + 1] - alo;
                for (int32_t j = 0; j < adeg && j < 32 && !found; j++) {
                    const int32_t x = l.slot_nb[alo + j];
                    if (x < l.n || l.ghost_src[x - l.n] != i || l.ghost_shift[x - l.n] != want) continue;
                    l.slot_edge[lo + q] = 2 * (l.edge_off[src] + __popc(l.edge_mask[src] & ((1u << j) - 1))) + 1;
                    found = true;
                }
            }
            bad |= !found;
        }
        const int32_t from_next = __shfl_sync(kAll, tri_before, first + (q + 1 < deg ? q + 1 : 0));
        if (tri < 0) tri = from_next;
        const int32_t before = __shfl_sync(kAll, tri, first + (q ? q - 1 : deg - 1));
        if (in) {
            bad |= tri < 0;
            l.slot_tri[lo + q] = tri;
        }
        if (own_edge) {
            const int32_t num = e0 + __popc(own_edges & ((1 << q) - 1));
            l.edge_l[num] = i;
            l.edge_r[num] = a;
            l.edge_ta[num] = before;
            l.edge_tb[num] = tri;
            l.slot_edge[lo + q] = 2 * num;
        }
        if (bad) report_bad(i);
    }
    report_counters(l);
}

inline int blocks(int64_t n, int b) { return (int)((n + b - 1) / b); }

// Blocks of 128 threads for a pass over every cell, four cells per warp,
// looping beyond `per SM` blocks on each of 152 SMs.  The update runs beside the
// FP64 stages of a sweep, which keep their pace as long as they hold most of
// the registers: at 1M cells a step and its read take 1.80 ms with 4 blocks
// per SM, 1.87 with 8, 1.88 with 16 and 2.09 with 2.  A split-precision sweep is
// over before the update, whose passes then count themselves: a step of 1M
// cells takes 1.03 ms with 4, 0.83 with 8, 0.82 with 16 and 0.93 with every
// block resident; of 640,000 cells 0.65, 0.55, 0.54 and 0.58; of 130,000 with 8
// and 16 0.221 and 0.207.
inline int pass_blocks(int64_t n, bool split)
{
    return std::max(1, std::min(blocks(8 * n, 128), kSMs * (split ? 16 : n >= (1 << 19) ? 4 : 8)));
}

}  // namespace

cudaError_t launch_lists(const MeshLists &l, bool alone, cudaStream_t st)
{
    if (l.n > 0) return launch_chained(k_mesh_lists, pass_blocks(l.n, alone), 128, st, l.n, l);
    return cudaSuccess;
}

cudaError_t MeshStore::reserve(int32_t n, const MeshSizes &z)
{
    const size_t i4 = sizeof(int32_t), N = (size_t)n, G = (size_t)z.ghosts + 1, T = (size_t)z.tris + 1;
    const size_t E = (size_t)z.edges + 1, S = (size_t)z.slots + 1;
    cudaError_t e = cudaSuccess;
    auto need = [&](DBuf &b, size_t bytes) {
        if (e == cudaSuccess) e = b.ensure(bytes);
    };
    need(cell_ptr, (N + 1) * i4);
    need(tri_off, (N + 1) * i4);
    need(edge_off, (N + 1) * i4);
    need(cell_order, N * i4);
    for (DBuf *b : {&slot_nb, &slot_tri, &slot_edge}) need(*b, S * i4);
    need(tri, 3 * T * i4);
    for (DBuf *b : {&edge_l, &edge_r, &edge_ta, &edge_tb}) need(*b, E * i4);
    for (DBuf *b : {&gx, &gy}) need(*b, G * sizeof(double));
    for (DBuf *b : {&ghost_src, &ghost_xf, &ghost_shift, &ghost_img}) need(*b, G * i4);
    if (e != cudaSuccess) release();
    return e;
}

void MeshStore::release()
{
    for (DBuf *b : {&cell_ptr, &slot_nb, &slot_tri, &slot_edge, &tri, &tri_off, &edge_off, &cell_order, &edge_l, &edge_r,
                    &edge_ta, &edge_tb, &gx, &gy, &ghost_src, &ghost_xf, &ghost_shift, &ghost_img})
        b->release();
}

MeshLists MeshStore::lists(int32_t n, int32_t periodic) const
{
    MeshLists l{};
    l.n = n;
    l.periodic = periodic;
    l.cell_ptr = cell_ptr.as<int32_t>();
    l.slot_nb = slot_nb.as<int32_t>();
    l.tri_off = tri_off.as<int32_t>();
    l.edge_off = edge_off.as<int32_t>();
    l.ghost_src = ghost_src.as<int32_t>();
    l.ghost_shift = ghost_shift.as<int32_t>();
    l.tri = tri.as<int32_t>();
    l.slot_tri = slot_tri.as<int32_t>();
    l.slot_edge = slot_edge.as<int32_t>();
    l.edge_l = edge_l.as<int32_t>();
    l.edge_r = edge_r.as<int32_t>();
    l.edge_ta = edge_ta.as<int32_t>();
    l.edge_tb = edge_tb.as<int32_t>();
    return l;
}

MeshOutput MeshStore::output(int32_t periodic) const
{
    MeshOutput o{};
    o.cell_ptr = cell_ptr.as<int32_t>();
    o.slot_nb = slot_nb.as<int32_t>();
    o.tri_off = tri_off.as<int32_t>();
    o.edge_off = edge_off.as<int32_t>();
    o.cell_order = cell_order.as<int32_t>();
    o.gx = gx.as<double>();
    o.gy = gy.as<double>();
    o.ghost_src = ghost_src.as<int32_t>();
    o.ghost_xf = ghost_xf.as<int32_t>();
    o.ghost_shift = ghost_shift.as<int32_t>();
    o.ghost_img = ghost_img.as<int32_t>();
    const size_t i4 = sizeof(int32_t);
    auto room = [](size_t entries) { return (int32_t)std::min<size_t>(entries, INT32_MAX / 4); };
    o.max.slots = room(std::min({slot_nb.cap, slot_tri.cap, slot_edge.cap}) / i4);
    o.max.edges = room(std::min({edge_l.cap, edge_r.cap, edge_ta.cap, edge_tb.cap}) / i4);
    o.max.tris = room(tri.cap / (3 * i4));
    o.max.ghosts = room(std::min({gx.cap / 8, gy.cap / 8, ghost_src.cap / i4, ghost_xf.cap / i4, ghost_shift.cap / i4,
                                  ghost_img.cap / i4}));
    o.lists = lists(0, periodic);
    return o;
}

cudaError_t MeshStream::create()
{
    // of the highest priority: its small kernels take the slots that blocks of
    // the sweep's large grids leave
    int least = 0, greatest = 0;
    cudaError_t e = cudaDeviceGetStreamPriorityRange(&least, &greatest);
    if (e == cudaSuccess) e = cudaStreamCreateWithPriority(&stream, cudaStreamNonBlocking, greatest);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&moved, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreate(&done);
    return e;
}

MeshStream::~MeshStream()
{
    if (stream) cudaStreamSynchronize(stream);
    if (moved) cudaEventDestroy(moved);
    if (done) cudaEventDestroy(done);
    if (stream) cudaStreamDestroy(stream);
}

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
    // stamps, which only ever grow, must start at zero
    const bool fresh = !(mark_.p && mark_.cap >= N * i4);
    MU_TRY(mark_.ensure(N * i4)); MU_TRY(info_.ensure(N * i4)); MU_TRY(extra_n_.ensure(N * i4));
    MU_TRY(list_[0].ensure(N * i4)); MU_TRY(list_[1].ensure(N * i4)); MU_TRY(heavy_.ensure(N * i4));
    MU_TRY(at_.ensure(N * i4));
    MU_TRY(ring_deg_.ensure(2 * R * i4)); MU_TRY(ring_ref_.ensure(2 * R * kMaxDeg * i4));
    MU_TRY(extra_.ensure(N * kMaxExtra * i4));
    if (sizes_.cap < N * 4) whole_ = true;
    MU_TRY(edge_mask_.ensure(N * 4)); MU_TRY(tri_mask_.ensure(N * 4));
    MU_TRY(sizes_.ensure(N * 4)); MU_TRY(images_.ensure(N * 2)); MU_TRY(ghost_off_.ensure((N + 1) * i4));
    MU_TRY(sums_.ensure((size_t)blocks(n, kWindow) * sizeof(int4)));
    // the counters, then the simulations' flags
    const size_t cb = sizeof(MeshUpdateCount) + (size_t)n_inst * i4;
    for (DBuf &c : count_)
        if (c.cap < cb) {
            MU_TRY(c.ensure(cb));
            MU_TRY(cudaMemsetAsync(c.p, 0, c.cap, st));
        }
    MU_TRY(host_.ensure(cb));
    if (fresh || stamp_ > (1 << 28)) {
        MU_TRY(cudaMemsetAsync(mark_.p, 0, mark_.cap, st));
        MU_TRY(cudaMemsetAsync(info_.p, 0, info_.cap, st));
        stamp_ = 0;
        told_ = true;
    }
    return cudaSuccess;
}

void MeshUpdater::release()
{
    for (DBuf *b : {&mark_, &list_[0], &list_[1], &heavy_, &info_, &at_, &ring_deg_, &ring_ref_, &extra_n_, &extra_,
                    &count_[0], &count_[1], &sizes_, &images_, &ghost_off_, &sums_, &edge_mask_, &tri_mask_})
        b->release();
    whole_ = told_ = true;
}

MeshUpdate MeshUpdater::params(const MeshArrays &a, const MeshOutput &o) const
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
    m.heavy = heavy_.as<int32_t>();
    m.ring_info = info_.as<int32_t>();
    m.ring_at = at_.as<int32_t>();
    m.max_rings = max_rings_;
    m.ring_deg = ring_deg_.as<int32_t>();
    m.ring_ref = ring_ref_.as<int32_t>();
    m.extra_n = extra_n_.as<int32_t>();
    m.extra = extra_.as<int32_t>();
    m.count = count_[0].as<MeshUpdateCount>();
    m.flags = reinterpret_cast<int32_t *>(m.count + 1);
    m.sizes = sizes_.as<uint32_t>();
    m.images = images_.as<uint16_t>();
    m.ghost_off = ghost_off_.as<int32_t>();
    m.edge_mask = edge_mask_.as<uint32_t>();
    m.tri_mask = tri_mask_.as<uint32_t>();
    m.out_ptr = o.cell_ptr;
    m.out_nb = o.slot_nb;
    m.tri_off = o.tri_off;
    m.edge_off = o.edge_off;
    m.cell_order = o.cell_order;
    m.gx = o.gx;
    m.gy = o.gy;
    m.gsrc = o.ghost_src;
    m.gxf = o.ghost_xf;
    m.gshift = o.ghost_shift;
    m.gimg = o.ghost_img;
    m.max_slots = o.max.slots;
    m.max_edges = o.max.edges;
    m.max_tris = o.max.tris;
    m.max_ghosts = o.max.ghosts;
    return m;
}

// rounds [first, last), then the new mesh if they settle it
cudaError_t MeshUpdater::launch_rounds(const MeshArrays &a, const MeshOutput &o, int first, int last, cudaStream_t st)
{
    const MeshUpdate m = params(a, o);
    // grids for the cells a step lists (a few per cent), looping beyond
    const int g = std::max(1, std::min(blocks(m.n, 16 * kListWarps), kSMs * 8));
    for (int r = first; r < last; r++) {
        if (r == 0) MU_TRY(launch_chained(k_mesh_recompute_light, g, kListBlock, st, m.n, m));
        MU_TRY(launch_chained(k_mesh_recompute, g, kListBlock, st, m.n, m, r));
        MU_TRY(launch_chained(k_mesh_check, g, kListBlock, st, m.n, m, r));
    }
    const int w = blocks(m.n, kWindow);
    MU_TRY(launch_chained(k_mesh_measure, w, kWindow, st, m.n, m, sums_.as<int4>(), (int32_t)(whole_ ? 1 : 0)));
    MU_TRY(launch_chained(k_mesh_offsets, w, kWindow, st, m.n, m, sums_.as<int4>(), (int32_t)last));
    MU_TRY(launch_chained(k_mesh_rings, pass_blocks(m.n, a.split), 128, st, m.n, m));
    MeshLists l = o.lists;
    l.n = a.n;
    l.cell_inst = a.cell_inst;
    l.inst = a.inst;
    l.cell_ptr = o.cell_ptr;
    l.slot_nb = o.slot_nb;
    l.tri_off = o.tri_off;
    l.edge_off = o.edge_off;
    l.ghost_src = o.ghost_src;
    l.ghost_shift = o.ghost_shift;
    l.edge_mask = m.edge_mask;
    l.tri_mask = m.tri_mask;
    l.ready = &m.count->ready;
    l.bad = &m.count->bad;
    l.flags = m.flags;
    l.next = count_[1].as<int32_t>();
    // (all of it: an update before the last may have had more simulations)
    l.next_words = (int32_t)(count_[1].cap / sizeof(int32_t));
    l.report = host_.as<int32_t>();
    l.done = &m.count->done;
    l.counters = count_[0].as<int32_t>();
    l.words = (int32_t)(sizeof(MeshUpdateCount) / sizeof(int32_t)) + a.n_inst;
    return launch_lists(l, a.split, st);
}

// The rounds launched before the host looks.  Most steps are settled by one; a
// second one's kernels are 5 us of empty launches in a step of 100 us (10,201
// cells), but the host's look and another launch of what follows are 50 us.
// So one round once kQuiet updates in a row needed no second.
constexpr int kQuiet = 8;

cudaError_t MeshUpdater::start(const MeshArrays &a, const MeshOutput &o, cudaStream_t st)
{
    const cudaError_t room = reserve(a.n, a.n_inst, st);
    if (room != cudaSuccess) {
        release();
        return room;
    }
    stamp_ += 16;
    static_assert(kMaxRounds + 1 < 16, "one update's stamps");
    // the counters cleared by the last update (or when they were allocated)
    std::swap(count_[0].p, count_[1].p);
    std::swap(count_[0].cap, count_[1].cap);
    // what an update that did not settle every cell it told of others left
    // behind: references in the numbering of the mesh it was started for
    if (told_) MU_TRY(cudaMemsetAsync(extra_n_.p, 0, extra_n_.cap, st));
    told_ = true;
    const MeshUpdate m = params(a, o);
    MU_TRY(launch_chained(k_mesh_verify, pass_blocks(a.n, a.split), kVerifyBlock, st, m.n, m));
    // (a warp per eight cells: steps of 10,201 cells took 105 us with one per
    // sixteen, 98 with this.  With the list passes at eight as well their FP64
    // tests slow the gradient of 4,096 cells, which runs beside them)
    const int open = std::max(1, std::min(blocks(a.n, 8 * kListWarps), kSMs * 8));
    MU_TRY(launch_chained(k_mesh_verify_open, open, kListBlock, st, m.n, m));
    last_round_ = quiet_ < kQuiet ? 2 : 1;
    return launch_rounds(a, o, 0, last_round_, st);
}

cudaError_t MeshUpdater::settle(const MeshArrays &a, const MeshOutput &o, MeshResult &result, cudaStream_t st)
{
    const MeshUpdateCount &c = *host_.as<MeshUpdateCount>();
    int r = last_round_;
    quiet_ = c.listed[1] > 0 ? 0 : std::min(quiet_ + 1, kQuiet);
    while (c.listed[r] > 0 && r < kMaxRounds) {
        const int to = std::min(r + 2, kMaxRounds);
        MU_TRY(launch_rounds(a, o, r, to, st));
        MU_TRY(cudaStreamSynchronize(st));
        r = to;
    }
    if (c.listed[r] > 0 && a.n_inst > 1) {
        const MeshUpdate m = params(a, o);
        k_mesh_give_up<<<64, 256, 0, st>>>(m, r);
        MU_TRY(cudaGetLastError());
        MU_TRY(cudaMemsetAsync(&m.count->listed[r], 0, sizeof(int32_t), st));
        MU_TRY(launch_rounds(a, o, r, r, st));
        MU_TRY(cudaStreamSynchronize(st));
    }
    result.sizes = MeshSizes{c.ghosts, c.tris, c.edges, c.slots};
    result.flagged = false;
    const int32_t *f = flags();
    for (int32_t k = 0; k < a.n_inst; k++) result.flagged |= f[k] != 0;
    const bool settled = c.listed[r] == 0 && c.slots >= 0 && c.slots <= INT32_MAX / 2;
    result.state = !settled ? MeshResult::kHost : c.ready ? MeshResult::kDone : MeshResult::kGrow;
    if (result.state == MeshResult::kGrow && a.n_inst == 1 && result.flagged) result.state = MeshResult::kHost;
    // (sizes of rings that were not kept are measured again)
    whole_ = result.state == MeshResult::kHost || result.flagged;
    told_ = whole_ || result.state == MeshResult::kGrow;
    last_round_ = r;
    return cudaSuccess;
}

cudaError_t MeshUpdater::again(const MeshArrays &a, const MeshOutput &o, MeshResult &result, cudaStream_t st)
{
    MU_TRY(launch_rounds(a, o, last_round_, last_round_, st));
    MU_TRY(cudaStreamSynchronize(st));
    return settle(a, o, result, st);
}

const int32_t *MeshUpdater::flags() const { return reinterpret_cast<const int32_t *>(host_.as<MeshUpdateCount>() + 1); }

}  // namespace rich
