// Update of a tessellation for moved points (a0): the predicates, frames,
// checks, sizes and ghosts of a cell, which the device kernels (meshupdate.cu)
// call, and the serial forms of verify, recompute_light, recompute and
// place_ring, which meshupdate_host.cpp runs.  Of those four the kernels are
// versions of their own, with lanes per ring slot or candidate; both are
// compared with the host builder (rich_device_update_check on the CPU,
// rich_mesh_check on the device).
//
// The mesh is the set of stars: every real cell's ring of Delaunay
// neighbours in counter-clockwise order.  Between steps the points move a
// fraction of a cell, and 0.01-2.6 % of the triangles change, so
//   verify    every cell checks its own star at the new positions: triangles
//             counter-clockwise, one turn, every edge locally Delaunay, the
//             circumdisks inside the ghost band; the cells of a failed check
//             are listed;
//   recompute a listed cell builds its star again by gift wrapping, at first
//             over its ring and the vertices the failed checks name (an edge
//             flip), else over the sources of its ring and of its neighbours'
//             rings (and their images, near a wall);
//   check     a new star's triangles must be in the rings of their other two
//             vertices, and a dropped neighbour must have dropped the cell;
//             where not, the cells involved are listed for another round and
//             told of the vertices they lack.
// This is star splaying (Shewchuk, "Star splaying: an algorithm for
// repairing Delaunay triangulations and convex hulls", 2005): stars that
// are all locally Delaunay and agree with each other form the Delaunay
// triangulation, which the symbolic tie-break makes unique, so the result is
// the host builder's mesh, ring for ring.  What the update does not handle (a
// circumdisk beyond the ghost band or a quarter of a periodic box; a listed cell
// of more than kMaxDeg neighbours, told vertices included, kMaxCand candidates
// or kMaxSources two-ring members; a cell of more than 32 neighbours beside one
// of up to eight; more than half the cells recomputed; rounds that do not
// converge; coordinates the exact predicates cannot hold) sets a flag of its
// simulation, and the caller builds that mesh on the host.
//
// Neighbours are references src * 16 + img: the image img = (a + 1) +
// 3 (b + 1), a, b in {-1, 0, 1}, of real cell src (4: the cell itself).  In a
// periodic box every neighbour is the source's image nearest to the cell,
// which holds while circumdisks are smaller than a quarter of the box
// (checked); across walls the image is part of the reference.
//
// Predicates: the sign of a determinant is taken from FP32 when it exceeds
// its error bound (FP64 runs at 1/64 of the FP32 rate on GB300; fewer than
// one edge in 10^4 goes on), else from FP64 with the host's bounds, else from
// exact integers (at once where periodic images are among the points).  This
// file must be compiled without floating-point contraction.
#pragma once

#include <cmath>
#include <cstdint>

#include "exactint.h"
#include "mesh.h"
#include "predicates.h"
#include "sweep.cuh"

namespace rich {

constexpr int kMaxDeg = 32;     // neighbours of a recomputed cell
constexpr int kLight = 16;      // candidates of recompute_light
constexpr int kMaxCand = 96;    // candidates of a recomputed cell
constexpr int kMaxSources = 256;  // cells of its neighbours' rings, repeats included (device)
constexpr int kMaxExtra = 8;    // vertices another cell can tell it of per round
constexpr int kMaxRounds = 12;  // rounds before the host takes over
constexpr int kMaxShift = 800;  // exponents to_float scales by

enum : int32_t {
    MU_FAR = 1,       // a circumdisk near or beyond the ghost band
    MU_SIZE = 2,      // too many candidates, neighbours or recomputed cells
    MU_STAR = 4,      // a star did not close (coincident points)
    MU_EXACT = 8,     // coordinates beyond the exact predicates' grid
    MU_IMAGE = 16,    // a neighbour image outside the ghost band
    MU_LISTS = 32,    // its rings do not agree with each other
    MU_ROUNDS = 64,   // stars that still disagreed after the last round
};

// Counters of one update (device memory, cleared at its start).
struct MeshUpdateCount {
    int32_t listed[kMaxRounds + 1];  // cells listed for each round
    int32_t open;                    // cells that FP32 could not verify
    int32_t heavy;                   // listed cells that recompute_light left
    int32_t overrides;               // cells recomputed so far
    int32_t slots, edges, tris, ghosts;
    int32_t ready;                   // the rounds are done and the new mesh fits its arrays
    int32_t bad;                     // the lists of the new mesh do not close
    int32_t done;                    // blocks that have written their lists
};

struct MeshUpdate {
    int32_t n, n_inst;
    const InstParams *inst;
    const int32_t *cell_inst;  // nullptr: one simulation
    const double *x, *y;       // new positions of the real cells
    // the mesh being updated
    const int32_t *cell_ptr, *slot_nb, *ghost_src, *ghost_img;
    // cells listed: stamp of the round a cell was last listed for, and the
    // rounds' lists (alternating).  Stamps grow from update to update, so
    // nothing is cleared between them.
    int32_t stamp;
    int32_t *mark, *list[2];  // (verify's undecided cells wait in list[1])
    int32_t *heavy;           // those of the first round that recompute_light left
    // recomputed stars: per cell (stamp << 2 | first << 1 | version) of its
    // last recomputation and its place, per place two versions of the ring
    int32_t *ring_info, *ring_at;
    int32_t max_rings;
    int32_t *ring_deg, *ring_ref;
    // vertices other cells found missing from a listed cell's star
    int32_t *extra_n, *extra;
    MeshUpdateCount *count;
    // MU_* of each simulation: a flagged one lists no more cells, and its
    // mesh is left to the host builder
    int32_t *flags;
    // per cell: owned edges, triangles, ghost images, degree (8 bits each)
    // and the mask of its images inside the ghost band
    uint32_t *sizes;
    uint16_t *images;
    // the updated mesh
    // (and for k_mesh_lists which of a ring's edges and triangles its cell owns)
    uint32_t *edge_mask, *tri_mask;
    int32_t *out_ptr, *out_nb, *tri_off, *edge_off, *ghost_off;
    double *gx, *gy;
    int32_t *gsrc, *gxf, *gshift, *gimg;
    int32_t *cell_order;
    int32_t max_slots, max_edges, max_tris, max_ghosts;
};

namespace mu {

#ifdef __CUDA_ARCH__
__device__ __forceinline__ int32_t a_exch(int32_t *p, int32_t v) { return atomicExch(p, v); }
__device__ __forceinline__ int32_t a_add(int32_t *p, int32_t v) { return atomicAdd(p, v); }
__device__ __forceinline__ void a_or(int32_t *p, int32_t v) { atomicOr(p, v); }
__device__ __forceinline__ int32_t vol(const int32_t *p) { return *(const volatile int32_t *)p; }
#else
inline int32_t a_exch(int32_t *p, int32_t v) { const int32_t o = *p; *p = v; return o; }
inline int32_t a_add(int32_t *p, int32_t v) { const int32_t o = *p; *p += v; return o; }
inline void a_or(int32_t *p, int32_t v) { *p |= v; }
inline int32_t vol(const int32_t *p) { return *p; }
#endif

// a < b by an order-preserving integer key (FP64 compares issue on the FP64 pipe)
RICH_HD inline bool less(double a, double b)
{
#ifdef __CUDA_ARCH__
    long long p = __double_as_longlong(a), q = __double_as_longlong(b);
    p ^= (p >> 63) & 0x7fffffffffffffffll;
    q ^= (q >> 63) & 0x7fffffffffffffffll;
    p = p == -1 ? 0 : p;
    q = q == -1 ? 0 : q;
    return p < q;
#else
    return a < b;
#endif
}

RICH_HD inline double image_coord(double v, double lo, double hi, int a, bool periodic)
{
    if (a == 0) return v;
    if (!periodic) return a < 0 ? (lo + lo) - v : (hi + hi) - v;
    return a > 0 ? v + (hi - lo) : v - (hi - lo);
}

// One cell's frame: its position, its simulation's box, and the power of two
// by which neighbour offsets are scaled for FP32 (a mean spacing becomes one
// to two).
struct Frame {
    const MeshUpdate *m;
    int32_t i;
    int32_t *flags;
    const InstParams *ip;
    double xi, yi;
    double x0, x1, y0, y1;  // box
    float half_x, half_y;   // half its sides (scaled)
    int32_t shift;
    float rlim2, rper2, reach;
    bool periodic;
};

RICH_HD inline int32_t inst_at(const MeshUpdate &m, int32_t i) { return m.cell_inst ? m.cell_inst[i] : 0; }

RICH_HD inline Frame frame_of(const MeshUpdate &m, int32_t i)
{
    const int32_t k = inst_at(m, i);
    const InstParams &ip = m.inst[k];
    Frame f;
    f.flags = m.flags + k;
    f.m = &m;
    f.i = i;
    f.ip = &ip;
    f.xi = m.x[i];
    f.yi = m.y[i];
    f.x0 = ip.x0; f.x1 = ip.x1; f.y0 = ip.y0; f.y1 = ip.y1;
    f.half_x = ip.half_x; f.half_y = ip.half_y;
    f.shift = ip.mesh_shift;
    f.rlim2 = ip.mesh_rlim2;
    f.rper2 = ip.mesh_rper2;
    f.reach = ip.mesh_reach;
    f.periodic = ip.boundary == 1;
    return f;
}

struct Point {
    double x, y;     // absolute position (as the host's ghost list has it)
    float fx, fy, l;  // scaled offset from the cell and its square
    int32_t ref;
};

// v 2^k (|k| <= kMaxShift) in FP32 with its mantissa cut to 24 bits, on the
// integer pipe (FP64 to FP32 conversions issue on the FP64 pipe); below FP32's
// normal range zero, above it infinite.  The scaling comes first, so that the
// range is about the point spacing whatever the box's units.
RICH_HD inline float to_float(double v, int32_t k)
{
#ifdef __CUDA_ARCH__
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const int e = (int)((hi >> 20) & 0x7ffu) + k;
    unsigned u = __funnelshift_l(lo, hi, 3) + ((unsigned)k << 23) - 0xc0000000u;
    u = e < 897 ? 0u : (e > 1150 ? 0x7f800000u : u);
    return __uint_as_float((u & 0x7fffffffu) | (hi & 0x80000000u));
#else
    const uint64_t b = exactint::bits_of(v);
    const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b;
    const int e = (int)((hi >> 20) & 0x7ffu) + k;
    unsigned u = ((hi << 3) | (lo >> 29)) + ((unsigned)k << 23) - 0xc0000000u;
    u = e < 897 ? 0u : (e > 1150 ? 0x7f800000u : u);
    u = (u & 0x7fffffffu) | (hi & 0x80000000u);
    float f;
    std::memcpy(&f, &u, 4);
    return f;
#endif
}

// the point of a reference; in a periodic box the source's nearest image
// (whatever image the reference names).  Neighbours are nearer than half the
// box by far (disk_ok), so FP32 decides which image that is.
RICH_HD inline Point point_of(const Frame &f, int32_t ref)
{
    const int32_t src = ref >> 4;
    Point p;
    p.x = f.m->x[src];
    p.y = f.m->y[src];
    p.ref = ref;
    if (!f.periodic) {
        const int32_t img = ref & 15;
        if (img != 4) {
            p.x = image_coord(p.x, f.x0, f.x1, img % 3 - 1, false);
            p.y = image_coord(p.y, f.y0, f.y1, img / 3 - 1, false);
        }
    }
    p.fx = to_float(p.x - f.xi, f.shift);
    p.fy = to_float(p.y - f.yi, f.shift);
    if (f.periodic) {
        int a = 0, b = 0;
        if (fabsf(p.fx) > f.half_x) {
            a = p.fx > 0.0f ? -1 : 1;
            p.x = image_coord(p.x, f.x0, f.x1, a, true);
            p.fx = to_float(p.x - f.xi, f.shift);
        }
        if (fabsf(p.fy) > f.half_y) {
            b = p.fy > 0.0f ? -1 : 1;
            p.y = image_coord(p.y, f.y0, f.y1, b, true);
            p.fy = to_float(p.y - f.yi, f.shift);
        }
        p.ref = src * 16 + (a + 1) + 3 * (b + 1);
    }
    p.l = p.fx * p.fx + p.fy * p.fy;
    return p;
}

// FP32 determinants of offsets, each offset within 2^-23 of its value (cut): a
// product of two is within 5 2^-24 and the cross product's error below 7 2^-24
// = 4.2e-7 of its permanent; |a|^2 is within 7 2^-24, and the in-circle sum
// within 18 2^-24 = 1.1e-6 of its permanent.  Below FP32's normal range errors
// are absolute instead: an offset is cut to zero from 2^-126, and products lose
// up to 2^-150 each.  With offsets up to r the two determinants are off by at
// most 4 r 2^-126 + 2^-149 and 24 r^3 2^-126 + 24 r^2 2^-150, below the floors
// for r up to 600 spacings; points 1e-11 spacings apart, whose in-circle sums
// are such numbers, are so left to FP64.
constexpr float kCrossBound = 1e-6f, kCrossFloor = 1e-30f;
constexpr float kCircleBound = 3e-6f, kCircleFloor = 1e-28f;
constexpr float kTinyTriangle = 1e-30f;  // 4 (twice its area)^2
RICH_HD inline float cross_error(float p, float q) { return kCrossBound * (fabsf(p) + fabsf(q)) + kCrossFloor; }
RICH_HD inline float circle_error(float al, float p1, float p2, float bl, float p3, float p4, float dl, float p5,
                                  float p6)
{
    return kCircleBound * (al * (fabsf(p1) + fabsf(p2)) + bl * (fabsf(p3) + fabsf(p4)) + dl * (fabsf(p5) + fabsf(p6))) +
           kCircleFloor;
}

#ifdef __CUDA_ARCH__
#define RICH_MU_SLOW __device__ __noinline__
#else
#define RICH_MU_SLOW inline
#endif

// orientation of a, b, c from FP64 with the host's bound, else exact
// (0 with MU_EXACT set when the integers cannot hold it)
RICH_MU_SLOW int orient_points(int32_t *flags, double ax, double ay, double bx, double by, double cx, double cy)
{
    const double l = (bx - ax) * (cy - ay), r = (by - ay) * (cx - ax);
    const double det = l - r, bound = kOrientBound * (fabs(l) + fabs(r));
    if (det > bound) return 1;
    if (-det > bound) return -1;
    if ((ax == bx && bx == cx) || (ay == by && by == cy)) return 0;
    const int s = exactint::orient_sign(ax, ay, bx, by, cx, cy);
    if (s == exactint::kUnknown) a_or(flags, MU_EXACT);
    return s == exactint::kUnknown ? 0 : s;
}

RICH_HD inline bool lex_less(double px, double py, double qx, double qy)
{
    return px < qx || (px == qx && py < qy);
}

// a <=> b for the exact sums p + q and r + s
RICH_HD inline int compare_sums(double p, double q, double r, double s, bool &known)
{
    const double s1 = p + q, v1 = s1 - p, e1 = (p - (s1 - v1)) + (q - v1);
    const double s2 = r + s, v2 = s2 - r, e2 = (r - (s2 - v2)) + (s - v2);
    const double d = (s1 - s2) + (e1 - e2);
    known = s1 == s2 || d != 0.0;
    return d > 0.0 ? 1 : (d < 0.0 ? -1 : 0);
}

// In-circle of four points that form two pairs of equal y (or x): the mirror
// images of two cells, and every square of a lattice.  The circle's centre is
// halfway between the other pair (r, s), so the power of d against that of
// its own partner m is (d - m)(d + m - r - s) along x: two exact sums instead
// of a 517-bit determinant.  1 inside, -1 outside, 0 on it, 2 when the points
// are no such pairs.
RICH_HD inline int circle_pairs(const double x[4], const double y[4])
{
    for (int k = 0; k < 3; k++) {  // the partner of d = point 3
        const int r = k == 0 ? 1 : 0, q = 3 - k - r;
        bool known = true;
        int s = 2;
        if (y[k] == y[3] && y[r] == y[q] && x[k] != x[3]) {
            s = compare_sums(x[3], x[k], x[r], x[q], known);
            s = x[3] > x[k] ? -s : s;
        } else if (x[k] == x[3] && x[r] == x[q] && y[k] != y[3]) {
            s = compare_sums(y[3], y[k], y[r], y[q], known);
            s = y[3] > y[k] ? -s : s;
        }
        if (s != 2 && known) return s;
    }
    return 2;
}

// in-circle of counter-clockwise a, b, c and d, likewise, with the symbolic
// tie-break of predicates.h: > 0 when d is inside
RICH_MU_SLOW int circle_points(int32_t *flags, double ax, double ay, double bx, double by, double cx, double cy,
                                 double dx, double dy)
{
    // (the pairs first: at walls nearly every slow test is one)
    const double px[4] = {ax, bx, cx, dx}, py[4] = {ay, by, cy, dy};
    int s = circle_pairs(px, py);
    if (s == 2) {
        const double adx = ax - dx, ady = ay - dy, bdx = bx - dx, bdy = by - dy, cdx = cx - dx, cdy = cy - dy;
        const double p1 = bdx * cdy, p2 = cdx * bdy, p3 = cdx * ady, p4 = adx * cdy, p5 = adx * bdy, p6 = bdx * ady;
        const double la = adx * adx + ady * ady, lb = bdx * bdx + bdy * bdy, lc = cdx * cdx + cdy * cdy;
        const double det = la * (p1 - p2) + lb * (p3 - p4) + lc * (p5 - p6);
        const double bound = kIncircleBound * (la * (fabs(p1) + fabs(p2)) + lb * (fabs(p3) + fabs(p4)) +
                                               lc * (fabs(p5) + fabs(p6)));
        // (infinities and NaNs fail the comparisons)
        if (det > bound && det < 1e300) return 1;
        if (-det > bound && -det < 1e300) return -1;
        s = exactint::incircle_sign(ax, ay, bx, by, cx, cy, dx, dy);
    }
    if (s == exactint::kUnknown) {
        a_or(flags, MU_EXACT);
        return 0;
    }
    if (s) return s;
    int k = 0;
    double mx = ax, my = ay;
    if (lex_less(bx, by, mx, my)) { k = 1; mx = bx; my = by; }
    if (lex_less(cx, cy, mx, my)) { k = 2; mx = cx; my = cy; }
    if (lex_less(dx, dy, mx, my)) { k = 3; }
    switch (k) {
    case 0: return orient_points(flags, bx, by, cx, cy, dx, dy);
    case 1: return -orient_points(flags, ax, ay, cx, cy, dx, dy);
    case 2: return orient_points(flags, ax, ay, bx, by, dx, dy);
    default: return -orient_points(flags, ax, ay, bx, by, cx, cy);
    }
}

// The slow predicates of images in a periodic box.  Every cell of a triangle
// or quadrilateral has to come to the same answer, but an image's coordinates
// are rounded, differently from each cell's own frame: near-ties (a drifting
// lattice is made of them) would then be decided differently on the two sides
// of the boundary.  So the images are taken exactly, as the host builder takes
// them: a cell's position and whole box sides.  (X, Y: the cells' positions;
// ref: the cell, a, b and for the in-circle test d.)
RICH_MU_SLOW int images_slow(int32_t *flags, const double *X, const double *Y, int32_t i, int32_t a, int32_t b,
                             int32_t d, double Lx, double Ly, bool circle)
{
    exactint::Images m;
    m.Lx = Lx;
    m.Ly = Ly;
    const int32_t ref[4] = {i * 16 + 4, a, b, d};
    for (int k = 0; k < 4; k++) {
        m.x[k] = X[ref[k] >> 4];
        m.y[k] = Y[ref[k] >> 4];
        m.kx[k] = (int8_t)((ref[k] & 15) % 3);
        m.ky[k] = (int8_t)((ref[k] & 15) / 3);
    }
    const int s = circle ? exactint::incircle_images(m) : exactint::orient_images(m);
    if (s != exactint::kUnknown) return s;
    a_or(flags, MU_EXACT);
    return 0;
}

// orientation of (cell, a, b)
RICH_HD inline int orient_slow(const Frame &f, const Point &a, const Point &b)
{
    if (f.periodic && ((a.ref & 15) != 4 || (b.ref & 15) != 4))
        return images_slow(f.flags, f.m->x, f.m->y, f.i, a.ref, b.ref, b.ref, f.x1 - f.x0, f.y1 - f.y0, false);
    return orient_points(f.flags, f.xi, f.yi, a.x, a.y, b.x, b.y);
}

// d against the circle of the counter-clockwise (cell, a, b)
RICH_HD inline int circle_slow(const Frame &f, const Point &a, const Point &b, const Point &d)
{
    if (f.periodic && ((a.ref & 15) != 4 || (b.ref & 15) != 4 || (d.ref & 15) != 4))
        return images_slow(f.flags, f.m->x, f.m->y, f.i, a.ref, b.ref, d.ref, f.x1 - f.x0, f.y1 - f.y0, true);
    return circle_points(f.flags, f.xi, f.yi, a.x, a.y, b.x, b.y, d.x, d.y);
}

// The same from references, for code that keeps no absolute positions: what is
// read again here costs it less than holding them (k_mesh_recompute of 50,625
// cells 22 us so, 25 with them; k_mesh_verify_open, which has them at hand, 24
// with them and 28 so).
RICH_MU_SLOW int refs_slow(int32_t *flags, const double *X, const double *Y, const InstParams *ip, int32_t i,
                           int32_t a, int32_t b, int32_t d, bool circle)
{
    const bool periodic = ip->boundary == 1;
    const int32_t ref[4] = {i * 16 + 4, a, b, d};
    if (periodic && ((a & 15) != 4 || (b & 15) != 4 || (d & 15) != 4))
        return images_slow(flags, X, Y, i, a, b, d, ip->x1 - ip->x0, ip->y1 - ip->y0, circle);
    double x[4], y[4];
    for (int k = 0; k < 4; k++) {
        const int img = ref[k] & 15;
        x[k] = X[ref[k] >> 4];
        y[k] = Y[ref[k] >> 4];
        if (img == 4) continue;
        x[k] = image_coord(x[k], ip->x0, ip->x1, img % 3 - 1, false);
        y[k] = image_coord(y[k], ip->y0, ip->y1, img / 3 - 1, false);
    }
    return circle ? circle_points(flags, x[0], y[0], x[1], y[1], x[2], y[2], x[3], y[3])
                  : orient_points(flags, x[0], y[0], x[1], y[1], x[2], y[2]);
}
RICH_HD inline int orient_slow(const Frame &f, int32_t a, int32_t b)
{
    return refs_slow(f.flags, f.m->x, f.m->y, f.ip, f.i, a, b, b, false);
}
RICH_HD inline int circle_slow(const Frame &f, int32_t a, int32_t b, int32_t d)
{
    return refs_slow(f.flags, f.m->x, f.m->y, f.ip, f.i, a, b, d, true);
}

// > 0 when d is inside the circumcircle of the counter-clockwise (cell, a, b).
// With offsets from the cell the determinant is
// -(|a|^2 (b x d) - |b|^2 (a x d) + |d|^2 (a x b)).
RICH_HD inline int incircle(const Frame &f, const Point &a, const Point &b, const Point &d)
{
    const float p1 = b.fx * d.fy, p2 = b.fy * d.fx, p3 = a.fx * d.fy, p4 = a.fy * d.fx, p5 = a.fx * b.fy,
                p6 = a.fy * b.fx;
    const float det = a.l * (p1 - p2) - b.l * (p3 - p4) + d.l * (p5 - p6);
    const float bound = circle_error(a.l, p1, p2, b.l, p3, p4, d.l, p5, p6);
    if (det > bound) return -1;
    if (-det > bound) return 1;
    return circle_slow(f, a, b, d);
}

// Whether a circumdisk of radius R about (ux, uy), from the cell, is inside the
// ghost band (all scaled).
RICH_HD inline bool disk_inside(const Frame &f, float ux, float uy, float R)
{
    const float lx = to_float(f.xi - f.x0, f.shift), rx = to_float(f.x1 - f.xi, f.shift);
    const float ly = to_float(f.yi - f.y0, f.shift), ry = to_float(f.y1 - f.yi, f.shift);
    return R - ux - lx <= f.reach && R + ux - rx <= f.reach && R - uy - ly <= f.reach && R + uy - ry <= f.reach;
}

// Whether the circumdisk of (cell, a, b) is certainly inside the ghost band
// (and, in a periodic box, smaller than a quarter of it).  A disk through
// the cell reaches past a wall by less than its diameter, so a radius below
// 0.48 bands is enough; larger disks are placed.  In FP32, with margins of
// 2 %; false for triangles of less than 2.5e-16 squared spacings, which the
// products underflow for (disk_ok_any takes them).
RICH_HD inline bool disk_ok(const Frame &f, const Point &a, const Point &b)
{
    const float cr = a.fx * b.fy - a.fy * b.fx;
    const float ex = a.fx - b.fx, ey = a.fy - b.fy;
    const float q = a.l * b.l * (ex * ex + ey * ey), c4 = 4.0f * cr * cr;
    if (!(c4 >= kTinyTriangle)) return false;
    if (q <= c4 * f.rlim2) return true;
    if (!(q <= c4 * f.rper2)) return false;
    const float i2 = 0.5f / cr;
    const float ux = (b.fy * a.l - a.fy * b.l) * i2, uy = (a.fx * b.l - b.fx * a.l) * i2;
    return disk_inside(f, ux, uy, sqrtf(ux * ux + uy * uy) * 1.001f);
}

// Circumcentre of (0, a, b) in FP64, all scaled (NaN where the cross product
// is of the size of its rounding).
RICH_MU_SLOW float2 centre_slow(double ax, double ay, double bx, double by, int32_t shift)
{
    const double s = exactint::pow2(shift);
    ax *= s;
    ay *= s;
    bx *= s;
    by *= s;
    const double l = ax * by, r = ay * bx, cr = l - r;
    float2 u = {NAN, NAN};
    if (fabs(cr) > 1e-12 * (fabs(l) + fabs(r))) {
        const double al = ax * ax + ay * ay, bl = bx * bx + by * by;
        u.x = to_float((by * al - ay * bl) / (cr + cr), 0);
        u.y = to_float((ax * bl - bx * al) / (cr + cr), 0);
    }
    return u;
}

// disk_ok for triangles of any size, in FP64 where FP32 has not the range.
RICH_HD inline bool disk_ok_any(const Frame &f, const Point &a, const Point &b)
{
    const float cr = a.fx * b.fy - a.fy * b.fx;
    if (4.0f * cr * cr >= kTinyTriangle) return disk_ok(f, a, b);
    const Point p = point_of(f, a.ref), q = point_of(f, b.ref);
    const float2 u = centre_slow(p.x - f.xi, p.y - f.yi, q.x - f.xi, q.y - f.yi, f.shift);
    const float R2 = u.x * u.x + u.y * u.y;
    return R2 <= f.rlim2 || (R2 <= f.rper2 && disk_inside(f, u.x, u.y, sqrtf(R2) * 1.001f));
}

// List a cell for the round of `stamp` (once).
RICH_HD inline void list_cell(const MeshUpdate &m, int32_t v, int32_t round)
{
    if (vol(m.flags + inst_at(m, v)) || vol(m.mark + v) == m.stamp + round || a_exch(m.mark + v, m.stamp + round) == m.stamp + round) return;
    m.list[round & 1][a_add(&m.count->listed[round], 1)] = v;
}

// Tell a listed cell v of reference r (in its own frame).
RICH_HD inline void tell_only(const MeshUpdate &m, int32_t v, int32_t r)
{
    const int32_t at = a_add(m.extra_n + v, 1);
    if (at < kMaxExtra) m.extra[(int64_t)v * kMaxExtra + at] = r;
}
RICH_HD inline void tell(const MeshUpdate &m, int32_t v, int32_t round, int32_t r)
{
    list_cell(m, v, round);
    tell_only(m, v, r);
}

RICH_HD inline int32_t base_ref(const MeshUpdate &m, int32_t q)
{
    return q < m.n ? q * 16 + 4 : m.ghost_src[q - m.n] * 16 + m.ghost_img[q - m.n];
}

// A cell's ring as another cell sees it.  While round `computing` is being
// recomputed its cells still show their previous star (-1: their latest).
struct Ring {
    const MeshUpdate *m;
    const int32_t *p;
    int32_t deg;
    bool base;
    RICH_HD int32_t operator[](int32_t k) const { return base ? base_ref(*m, p[k]) : p[k]; }
};

RICH_HD inline Ring ring_of(const MeshUpdate &m, int32_t v, int32_t computing)
{
    const int32_t info = vol(m.ring_info + v);
    bool base = (info >> 2) < m.stamp;
    int ver = info & 1;
    if (!base && computing >= 0 && (info >> 2) == m.stamp + computing) {
        if (info & 2) base = true;
        else ver ^= 1;
    }
    Ring r;
    r.m = &m;
    r.base = base;
    if (base) {
        r.p = m.slot_nb + m.cell_ptr[v];
        r.deg = m.cell_ptr[v + 1] - m.cell_ptr[v];
    } else {
        const int32_t at = 2 * m.ring_at[v] + ver;
        r.p = m.ring_ref + (int64_t)at * kMaxDeg;
        r.deg = m.ring_deg[at];
    }
    return r;
}

// Whether an image of a ring member (or of the cell) across the walls that
// the ring meets lies in the circle of (cell, b, d).
RICH_HD inline bool image_inside(const Frame &f, const int32_t *nb, int32_t deg, const Point &b, const Point &d)
{
    uint32_t imgs = 0;
    for (int32_t k = 0; k < deg; k++) imgs |= 1u << (base_ref(*f.m, nb[k]) & 15);
    for (int img = 0; img < 9; img++) {
        if (img == 4 || !(imgs >> img & 1)) continue;
        for (int32_t k = -1; k < deg; k++) {
            const int32_t r = (k < 0 ? f.i : base_ref(*f.m, nb[k]) >> 4) * 16 + img;
            if (r == b.ref || r == d.ref) continue;
            if (incircle(f, b, d, point_of(f, r)) > 0) return true;
        }
    }
    return false;
}

// ---- the bodies --------------------------------------------------------------

// The edge from a cell to b between its neighbours a and d is not locally
// Delaunay: its end loses it, and a and d may gain each other.
RICH_HD inline void list_bad(const MeshUpdate &m, bool periodic, int32_t a, int32_t b, int32_t d)
{
    list_cell(m, b >> 4, 0);
    // (across a wall a reference holds in the frame of a cell itself only)
    if (periodic || (a & 15) == 4) tell(m, a >> 4, 0, d);
    else list_cell(m, a >> 4, 0);
    if (periodic || (d & 15) == 4) tell(m, d >> 4, 0, a);
    else list_cell(m, d >> 4, 0);
}

// Cell i's star at the new positions.  With kFast the predicates stop at
// FP32 and a star that they cannot decide is reported (true) instead, for a
// second call without: the pass over every cell then holds no FP64 or exact
// code, and its registers leave room for twice the warps.
template <bool kFast> RICH_HD inline bool verify(const MeshUpdate &m, int32_t i)
{
    const Frame f = frame_of(m, i);
    const int32_t lo = m.cell_ptr[i], deg = m.cell_ptr[i + 1] - lo;
    const int32_t *nb = m.slot_nb + lo;
    Point a = point_of(f, base_ref(m, nb[deg - 2])), b = point_of(f, base_ref(m, nb[deg - 1]));
    // (a x b: the orientation of the triangle before the first)
    float cab = a.fx * b.fy - a.fy * b.fx;
    int turns = 0;
    bool self = false, open = false;
    for (int32_t k = 0; k < deg; k++) {
        const int32_t ref = base_ref(m, nb[k]);
        const Point d = point_of(f, ref);
        const float p = b.fx * d.fy, q = b.fy * d.fx, cbd = p - q;
        bool bad = false;
        if (!(cbd > cross_error(p, q))) {
            if (kFast) open = true;
            else bad = orient_slow(f, b, d) <= 0;
        }
        const float p3 = a.fx * d.fy, p4 = a.fy * d.fx, p5 = a.fx * b.fy, p6 = a.fy * b.fx;
        const float det = a.l * cbd - b.l * (p3 - p4) + d.l * cab;
        const float bound = circle_error(a.l, p, q, b.l, p3, p4, d.l, p5, p6);
        if (!(det > bound)) {
            if (-det > bound) bad = true;
            else if (kFast) open = true;
            else if (!bad) bad = circle_slow(f, a, b, d) >= 0;
        }
        // both other vertices images across a wall: what lies beyond their
        // edge is the image of a cell around this one, and no star of a cell
        // tests it
        if (!f.periodic && (b.ref & 15) != 4 && (d.ref & 15) != 4) {
            if (kFast) open = true;
            else if (!bad) bad = image_inside(f, nb, deg, b, d);
        }
        if (bad && !(kFast && open)) {
            list_bad(m, f.periodic, a.ref, b.ref, d.ref);
            self = true;
        }
        // another image than the mesh had, or a disk near the band's edge:
        // this cell alone
        if (d.ref != ref || !(kFast ? disk_ok(f, b, d) : disk_ok_any(f, b, d))) self = true;
        turns += (b.fy < 0.0f && d.fy >= 0.0f) ? 1 : 0;
        a = b;
        b = d;
        cab = cbd;
    }
    if (kFast && open) return true;
    if (self || turns != 1) list_cell(m, i, 0);
    return false;
}

// Cell i's star from its ring and the vertices it was told of, in FP32: what
// an edge flip asks for, and with it nearly every listed cell.  Returns
// false, with nothing written, where that does not settle it (a cell at a wall, a
// predicate beyond FP32, a large star or disk): recompute then.  (Serial; the
// device's k_mesh_recompute_light takes a lane per candidate.)
inline bool recompute_light(const MeshUpdate &m, int32_t i, int32_t round)
{
    int32_t ref[kLight];
    float fx[kLight], fy[kLight];

    const Frame f = frame_of(m, i);
    const Ring own = ring_of(m, i, round);
    const int32_t ne = m.extra_n[i];
    if (own.deg + ne > kLight || ne > kMaxExtra) return false;
    int nc = 0, near = 0;
    float lmin = 0.0f;
    for (int32_t k = 0; k < own.deg + ne; k++) {
        const int32_t r = k < own.deg ? own[k] : m.extra[(int64_t)i * kMaxExtra + (k - own.deg)];
        if (!f.periodic && (r & 15) != 4) return false;
        if ((r >> 4) == i) return false;
        bool have = false;
        for (int c = 0; c < nc; c++) have |= (ref[c] >> 4) == (r >> 4);
        if (have) continue;
        const Point p = point_of(f, r);
        ref[nc] = p.ref;
        fx[nc] = p.fx;
        fy[nc] = p.fy;
        if (nc == 0 || p.l < lmin) {
            lmin = p.l;
            near = nc;
        }
        nc++;
    }
    // (the nearest candidate in FP32 is a neighbour unless another lies
    // within a thousandth of its distance of it; the wrapping then does not
    // close)
    uint64_t out = 0;  // candidates in ring order, 4 bits each
    int deg = 0, last = near, turns = 0;
    do {
        if (deg == 16) return false;
        out |= (uint64_t)last << (4 * deg);
        deg++;
        Point a;
        a.fx = fx[last];
        a.fy = fy[last];
        a.l = a.fx * a.fx + a.fy * a.fy;
        int best = -1;
        Point b;
        for (int k = 0; k < nc; k++) {
            if (k == last) continue;
            Point d;
            d.fx = fx[k];
            d.fy = fy[k];
            const float p3 = a.fx * d.fy, p4 = a.fy * d.fx, c = p3 - p4, cb = cross_error(p3, p4);
            if (-c > cb) continue;
            if (!(c > cb)) return false;
            d.l = d.fx * d.fx + d.fy * d.fy;
            if (best >= 0) {
                const float p1 = b.fx * d.fy, p2 = b.fy * d.fx, p5 = a.fx * b.fy, p6 = a.fy * b.fx;
                const float det = a.l * (p1 - p2) - b.l * c + d.l * (p5 - p6);
                const float bound = circle_error(a.l, p1, p2, b.l, p3, p4, d.l, p5, p6);
                if (det > bound) continue;
                if (!(-det > bound)) return false;
            }
            best = k;
            b = d;
        }
        if (best < 0 || !disk_ok(f, a, b)) return false;
        turns += (a.fy < 0.0f && b.fy >= 0.0f) ? 1 : 0;
        last = best;
    } while (last != near);
    if (deg < 3 || turns != 1) return false;
    const int32_t info = m.ring_info[i];
    const bool fresh = (info >> 2) < m.stamp;
    int32_t at, ver = 0;
    if (fresh) {
        at = a_add(&m.count->overrides, 1);
        if (at >= m.max_rings) {
            a_or(f.flags, MU_SIZE);
            return true;
        }
        m.ring_at[i] = at;
    } else {
        at = m.ring_at[i];
        ver = (info & 1) ^ 1;
    }
    int32_t *dst = m.ring_ref + (int64_t)(2 * at + ver) * kMaxDeg;
    for (int k = 0; k < deg; k++) dst[k] = ref[(int)(out >> (4 * k) & 15)];
    m.ring_deg[2 * at + ver] = deg;
    m.ring_info[i] = (m.stamp + round) << 2 | (fresh ? 2 : 0) | ver;
    m.extra_n[i] = 0;
    return true;
}

// Cell i's star built again from the candidates around it (serial; the device
// runs the same steps with a warp per cell, see k_mesh_recompute).
RICH_HD inline void recompute(const MeshUpdate &m, int32_t i, int32_t round)
{
    const Frame f = frame_of(m, i);
    int32_t src[kMaxCand];
    int ns = 0;
    uint32_t imgs = 1u << 4;
    bool full = false;
    auto add = [&](int32_t s) {
        for (int k = 0; k < ns; k++)
            if (src[k] == s) return;
        if (ns == kMaxCand) full = true;
        else src[ns++] = s;
    };
    // sources of the ring and of what others reported, then of their rings
    const Ring own = ring_of(m, i, round);
    for (int32_t k = 0; k < own.deg; k++) {
        const int32_t r = own[k];
        imgs |= 1u << (r & 15);
        if ((r >> 4) != i) add(r >> 4);
    }
    const int32_t told = m.extra_n[i], ne = told < kMaxExtra ? told : kMaxExtra;
    m.extra_n[i] = 0;
    for (int32_t k = 0; k < ne; k++) {
        const int32_t r = m.extra[(int64_t)i * kMaxExtra + k];
        imgs |= 1u << (r & 15);
        if ((r >> 4) != i) add(r >> 4);
    }
    const int first = ns;
    for (int k = 0; k < first; k++) {
        const Ring r = ring_of(m, src[k], round);
        for (int32_t j = 0; j < r.deg; j++) {
            const int32_t q = r[j];
            imgs |= 1u << (q & 15);
            if ((q >> 4) != i) add(q >> 4);
        }
    }
    // the candidates: nearest images, or every source's images across the
    // walls that any of these rings meets (the cell's own images too)
    int32_t ref[kMaxCand];
    float fx[kMaxCand], fy[kMaxCand], fl[kMaxCand];
    int nc = 0;
    int near = -1;
    double dmin = 0.0;
    auto put = [&](int32_t r) {
        if (nc == kMaxCand) {
            full = true;
            return;
        }
        const Point p = point_of(f, r);
        ref[nc] = p.ref;
        fx[nc] = p.fx;
        fy[nc] = p.fy;
        fl[nc] = p.l;
        const double dx = p.x - f.xi, dy = p.y - f.yi, d2 = dx * dx + dy * dy;
        if (near < 0 || d2 < dmin) {
            near = nc;
            dmin = d2;
        }
        nc++;
    };
    for (int k = 0; k < ns; k++) put(src[k] * 16 + 4);
    if (!f.periodic && imgs != 1u << 4)
        for (int img = 0; img < 9; img++) {
            if (img == 4 || !(imgs >> img & 1)) continue;
            put(i * 16 + img);
            for (int k = 0; k < ns; k++) put(src[k] * 16 + img);
        }
    if (full || nc < 3) {
        a_or(f.flags, MU_SIZE);
        return;
    }
    auto point = [&](int k) {
        Point p;
        p.fx = fx[k];
        p.fy = fy[k];
        p.l = fl[k];
        p.ref = ref[k];
        return p;
    };
    // (FP32 in-circle: with offsets from the cell, d is inside the circle of
    // the counter-clockwise (cell, a, b) when |a|^2 (b x d) - |b|^2 (a x d) +
    // |d|^2 (a x b) < 0)
    // gift wrapping from the nearest candidate (always a neighbour): the next
    // one is the point to the left of the last whose circle with the cell and
    // the last is empty
    int32_t out[kMaxDeg];
    int deg = 0, last = near, turns = 0;
    bool bad = false;
    do {
        if (deg == kMaxDeg) {
            bad = true;
            break;
        }
        out[deg++] = ref[last];
        const Point a = point(last);
        int best = -1;
        for (int k = 0; k < nc; k++) {
            if (k == last) continue;
            const float p = a.fx * fy[k], q = a.fy * fx[k], c = p - q;
            const float cb = cross_error(p, q);
            bool left = c > cb;
            if (!left && !(-c > cb)) left = orient_slow(f, ref[last], ref[k]) > 0;
            if (!left) continue;
            if (best < 0) {
                best = k;
                continue;
            }
            const Point b = point(best);
            const float p1 = b.fx * fy[k], p2 = b.fy * fx[k], p5 = a.fx * b.fy, p6 = a.fy * b.fx;
            const float det = a.l * (p1 - p2) - b.l * c + fl[k] * (p5 - p6);
            const float bound = circle_error(a.l, p1, p2, b.l, p, q, fl[k], p5, p6);
            if (det > bound) continue;
            if (-det > bound || circle_slow(f, ref[last], ref[best], ref[k]) > 0) best = k;
        }
        if (best < 0) {
            bad = true;
            break;
        }
        if (!disk_ok_any(f, a, point(best))) a_or(f.flags, MU_FAR);
        turns += (a.fy < 0.0f && fy[best] >= 0.0f) ? 1 : 0;
        last = best;
    } while (last != near);
    if (bad || deg < 3 || turns != 1) {
        a_or(f.flags, MU_STAR);
        return;
    }
    // into the version that no other cell reads in this round
    const int32_t info = m.ring_info[i];
    const bool fresh = (info >> 2) < m.stamp;
    int32_t at, ver;
    if (fresh) {
        at = a_add(&m.count->overrides, 1);
        if (at >= m.max_rings) {
            a_or(f.flags, MU_SIZE);
            return;
        }
        m.ring_at[i] = at;
        ver = 0;
    } else {
        at = m.ring_at[i];
        ver = (info & 1) ^ 1;
    }
    int32_t *dst = m.ring_ref + (int64_t)(2 * at + ver) * kMaxDeg;
    for (int k = 0; k < deg; k++) dst[k] = out[k];
    m.ring_deg[2 * at + ver] = deg;
    m.ring_info[i] = (m.stamp + round) << 2 | (fresh ? 2 : 0) | ver;
}

// whether the ring of v has r followed by q (by source in a periodic box)
RICH_HD inline bool has_pair(const MeshUpdate &m, bool periodic, int32_t v, int32_t r, int32_t q)
{
    const Ring g = ring_of(m, v, -1);
    int32_t prev = g[g.deg - 1];
    for (int32_t k = 0; k < g.deg; k++) {
        const int32_t cur = g[k];
        if (periodic ? ((prev >> 4) == (r >> 4) && (cur >> 4) == (q >> 4)) : (prev == r && cur == q)) return true;
        prev = cur;
    }
    return false;
}

// The new star of cell i against its neighbours' rings: slot k's triangle,
// and slot k of the star it replaced (the device's lanes take one k each).
RICH_HD inline bool recomputed(const MeshUpdate &m, int32_t i, int32_t round)
{
    return (m.ring_info[i] >> 2) == m.stamp + round;  // else a flag is set
}

RICH_HD inline void check_triangle(const MeshUpdate &m, bool periodic, const Ring &g, int32_t i, int32_t round,
                                   int32_t k)
{
    const int32_t me = i * 16 + 4, a = g[k ? k - 1 : g.deg - 1], b = g[k];
    // the triangle (i, a, b) in the rings of a and b (the cells themselves,
    // not their images across a wall)
    if ((periodic || (a & 15) == 4) && !has_pair(m, periodic, a >> 4, b, me)) {
        tell(m, a >> 4, round + 1, b);
        tell(m, a >> 4, round + 1, me);
        list_cell(m, i, round + 1);
    }
    if ((periodic || (b & 15) == 4) && !has_pair(m, periodic, b >> 4, me, a)) {
        tell(m, b >> 4, round + 1, me);
        tell(m, b >> 4, round + 1, a);
        list_cell(m, i, round + 1);
    }
}

// a neighbour of the previous star that the new one dropped must have dropped
// the cell
RICH_HD inline void check_dropped(const MeshUpdate &m, bool periodic, const Ring &g, const Ring &old, int32_t i,
                                  int32_t round, int32_t k)
{
    const int32_t me = i * 16 + 4, r = old[k];
    if ((r >> 4) == i || (!periodic && (r & 15) != 4)) return;
    for (int32_t j = 0; j < g.deg; j++)
        if (periodic ? (g[j] >> 4) == (r >> 4) : g[j] == r) return;
    const Ring o = ring_of(m, r >> 4, -1);
    for (int32_t j = 0; j < o.deg; j++)
        if (periodic ? (o[j] >> 4) == i : o[j] == me) {
            list_cell(m, r >> 4, round + 1);
            return;
        }
}

// The images of point (x, y) inside the ghost band, in the host builder's
// order (bit img of the mask; make_ghosts).
RICH_HD inline uint32_t image_mask(const InstParams &ip, double x, double y)
{
    if (less(ip.in_x0, x) && less(x, ip.in_x1) && less(ip.in_y0, y) && less(y, ip.in_y1)) return 0;
    const bool per = ip.boundary == 1;
    const double lox = ip.x0 - ip.band, hix = ip.x1 + ip.band, loy = ip.y0 - ip.band, hiy = ip.y1 + ip.band;
    uint32_t ox = 0, oy = 0;
    for (int a = -1; a <= 1; a++) {
        const double X = image_coord(x, ip.x0, ip.x1, a, per), Y = image_coord(y, ip.y0, ip.y1, a, per);
        if (!(X < lox || X > hix)) ox |= 1u << (a + 1);
        if (!(Y < loy || Y > hiy)) oy |= 1u << (a + 1);
    }
    if (!((ox | oy) & 5u)) return 0;
    uint32_t mask = 0;
    for (int b = 0; b < 3; b++)
        if (oy >> b & 1) mask |= ox << (3 * b);
    return mask & ~(1u << 4);
}

RICH_HD inline int popcount(uint32_t v)
{
#ifdef __CUDA_ARCH__
    return __popc(v);
#else
    return __builtin_popcount(v);
#endif
}

// position of image img among the images of `mask` in the host's order:
// a (x) outer, b (y) inner
RICH_HD inline int image_rank(uint32_t mask, int img)
{
    const int a = img % 3, b = img / 3;
    int r = 0;
    for (int q = 0; q < 9; q++) {
        if (!(mask >> q & 1)) continue;
        const int qa = q % 3, qb = q / 3;
        r += (qa < a || (qa == a && qb < b)) ? 1 : 0;
    }
    return r;
}

// A ring's degree, owned edges and owned triangles (8 bits each).
RICH_HD inline uint32_t ring_sizes(const MeshUpdate &m, bool periodic, int32_t i, const Ring &g)
{
    uint32_t ne = 0, nt = 0;
    const int32_t prev = g[g.deg - 1];
    bool prev_up = (prev & 15) != 4 || (prev >> 4) > i;
    for (int32_t k = 0; k < g.deg; k++) {
        const int32_t r = g[k];
        const bool real = (r & 15) == 4, up = !real || (r >> 4) > i;
        ne += real || periodic ? (r >> 4) > i : 1;
        nt += (prev_up && up) ? 1 : 0;
        prev_up = up;
    }
    if (g.deg > 255) a_or(m.flags + inst_at(m, i), MU_SIZE);
    return (uint32_t)(g.deg & 255) | ne << 8 | nt << 16;
}

// The cell's images inside the ghost band, counted into its sizes.
RICH_HD inline uint32_t count_images(const MeshUpdate &m, int32_t i, uint32_t ring_part)
{
    const uint32_t mask = image_mask(m.inst[inst_at(m, i)], m.x[i], m.y[i]);
    m.images[i] = (uint16_t)mask;
    return (ring_part & 0xffffffu) | (uint32_t)popcount(mask) << 24;
}

// The cell's degree, owned edges and triangles, and ghost images.
RICH_HD inline uint32_t measure(const MeshUpdate &m, int32_t i)
{
    const bool periodic = m.inst[inst_at(m, i)].boundary == 1;
    return m.sizes[i] = count_images(m, i, ring_sizes(m, periodic, i, ring_of(m, i, -1)));
}

// The ghosts of cell i, from ghost_off[i] on.
RICH_HD inline void place_ghosts(const MeshUpdate &m, int32_t i)
{
    const uint32_t mask = m.images[i];
    if (!mask) return;
    const InstParams &ip = m.inst[inst_at(m, i)];
    const bool per = ip.boundary == 1;
    int32_t k = m.ghost_off[i];
    for (int a = -1; a <= 1; a++)
        for (int b = -1; b <= 1; b++) {
            const int img = (a + 1) + 3 * (b + 1);
            if (!(mask >> img & 1)) continue;
            m.gx[k] = image_coord(m.x[i], ip.x0, ip.x1, a, per);
            m.gy[k] = image_coord(m.y[i], ip.y0, ip.y1, b, per);
            m.gsrc[k] = i;
            m.gxf[k] = per ? 0 : ((a ? XF_MIRROR_X : 0) | (b ? XF_MIRROR_Y : 0));
            m.gshift[k] = per ? img : 4;
            m.gimg[k] = img;
            k++;
        }
}

// the updated mesh's point of a reference in cell i's ring
RICH_HD inline int32_t point_id(const MeshUpdate &m, int32_t i, int32_t r)
{
    const int32_t src = r >> 4, img = r & 15;
    if (img == 4) return src;
    const uint32_t mask = m.images[src];
    if (!(mask >> img & 1)) {
        a_or(m.flags + inst_at(m, i), MU_IMAGE);
        a_or(&m.count->bad, 1);
        return src;
    }
    return m.n + m.ghost_off[src] + image_rank(mask, img);
}

// Cell i's ring with this mesh's point ids, from its smallest neighbour on
// (serial; the device's k_mesh_rings takes eight lanes per cell).
RICH_HD inline void place_ring(const MeshUpdate &m, int32_t i)
{
    const Ring g = ring_of(m, i, -1);
    int32_t *dst = m.out_nb + m.out_ptr[i];
    int32_t best = INT32_MAX, at = 0;
    for (int32_t k = 0; k < g.deg; k++) {
        const int32_t id = point_id(m, i, g[k]);
        if (id < best) {
            best = id;
            at = k;
        }
    }
    for (int32_t k = 0; k < g.deg; k++) dst[k] = point_id(m, i, g[at + k < g.deg ? at + k : at + k - g.deg]);
}

}  // namespace mu

// The update's constants in a simulation's parameters (host): its ghost band
// as build_host_mesh takes it first, and the FP32 limits on circumdisks.
void mesh_params(const BoxConfig &box, int32_t n, InstParams &ip);

// The update of `mesh` (a build_host_mesh result, or this function's) for
// new points by the serial forms above, on the host.  Returns 1, or
// 0 with `flags` set when the host builder has to take the mesh.
int mesh_update_serial(const BoxConfig &box, int32_t n, const double *x, const double *y, HostMesh &mesh,
                       int32_t &flags, int32_t &rounds, int32_t &recomputed);

}  // namespace rich
