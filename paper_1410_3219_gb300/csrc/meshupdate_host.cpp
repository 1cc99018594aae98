// Host side of the mesh update of meshupdate.h: its constants, and a run of its
// serial forms that the tests compare with the host builder.
#include "meshupdate.h"

#include <algorithm>
#include <cmath>
#include <vector>

namespace rich {

void mesh_params(const BoxConfig &box, int32_t n, InstParams &ip)
{
    const double Lx = box.x1 - box.x0, Ly = box.y1 - box.y0, lmin = std::min(Lx, Ly);
    // the first band build_host_mesh tries, and the margin of make_ghosts
    const double h = std::sqrt(Lx * Ly / std::max(n, 1));
    const double w = std::min(5.0 * h, lmin);
    const double margin = 1e-9 * (std::fabs(box.x0) + std::fabs(box.x1) + std::fabs(box.y0) + std::fabs(box.y1) + w);
    // the power of two that scales a mean spacing to [1, 2)
    ip.mesh_shift = h > 0.0 && std::isfinite(h) ? std::max(-kMaxShift, std::min(kMaxShift, -std::ilogb(h))) : 0;
    const double scale = exactint::pow2(ip.mesh_shift);
    ip.half_x = (float)(0.5 * Lx * scale);
    ip.half_y = (float)(0.5 * Ly * scale);
    ip.band = w;
    ip.in_x0 = box.x0 + w + margin;
    ip.in_x1 = box.x1 - w - margin;
    ip.in_y0 = box.y0 + w + margin;
    ip.in_y1 = box.y1 - w - margin;
    const double rl = 0.48 * w * scale, rp = box.boundary == 1 ? 0.24 * lmin * scale : 1e18;
    ip.mesh_rlim2 = (float)(std::min(rl, rp) * std::min(rl, rp));
    ip.mesh_rper2 = (float)(rp * rp);
    ip.mesh_reach = (float)(0.98 * w * scale);
}

int mesh_update_serial(const BoxConfig &box, int32_t n, const double *x, const double *y, HostMesh &mesh, int32_t &flags,
                       int32_t &rounds, int32_t &recomputed)
{
    InstParams ip{};
    ip.boundary = box.boundary;
    ip.x0 = box.x0; ip.x1 = box.x1; ip.y0 = box.y0; ip.y1 = box.y1;
    mesh_params(box, n, ip);
    MeshUpdate m{};
    MeshUpdateCount cnt{};
    m.n = n;
    m.n_inst = 1;
    m.inst = &ip;
    m.x = x;
    m.y = y;
    m.cell_ptr = mesh.cell_ptr.data();
    m.slot_nb = mesh.slot_nb.data();
    m.ghost_src = mesh.ghost_src.data();
    m.ghost_img = mesh.ghost_img.data();
    m.stamp = 1;
    m.max_rings = n;
    std::vector<int32_t> mark(n, 0), l0(n), l1(n), info(n, 0), at(n), deg(2 * (size_t)n), ref(2 * (size_t)n * kMaxDeg);
    std::vector<int32_t> en(n, 0), ex((size_t)n * kMaxExtra);
    std::vector<uint32_t> sizes(n);
    std::vector<uint16_t> images(n);
    m.mark = mark.data();
    m.list[0] = l0.data();
    m.list[1] = l1.data();
    m.ring_info = info.data();
    m.ring_at = at.data();
    m.ring_deg = deg.data();
    m.ring_ref = ref.data();
    m.extra_n = en.data();
    m.extra = ex.data();
    m.count = &cnt;
    flags = 0;
    m.flags = &flags;
    m.sizes = sizes.data();
    m.images = images.data();
    for (int32_t i = 0; i < n; i++)
        if (mu::verify<true>(m, i)) m.list[1][cnt.open++] = i;
    for (int32_t k = 0; k < cnt.open; k++) mu::verify<false>(m, m.list[1][k]);
    rounds = 0;
    recomputed = 0;
    for (; rounds < kMaxRounds && cnt.listed[rounds] > 0; rounds++) {
        for (int32_t k = 0; k < cnt.listed[rounds]; k++) {
            const int32_t i = m.list[rounds & 1][k];
            if (rounds == 0 && mu::recompute_light(m, i, rounds)) continue;
            mu::recompute(m, i, rounds);
        }
        for (int32_t k = 0; k < cnt.listed[rounds]; k++) {
            const int32_t i = m.list[rounds & 1][k];
            if (!mu::recomputed(m, i, rounds)) continue;
            const mu::Ring g = mu::ring_of(m, i, -1), old = mu::ring_of(m, i, rounds);
            for (int32_t t = 0; t < g.deg; t++) mu::check_triangle(m, box.boundary == 1, g, i, rounds, t);
            for (int32_t t = 0; t < old.deg; t++) mu::check_dropped(m, box.boundary == 1, g, old, i, rounds, t);
        }
        recomputed += cnt.listed[rounds];
    }
    if (flags || cnt.listed[rounds] > 0) return 0;
    HostMesh out;
    out.n = n;
    out.cell_ptr.resize(n + 1);
    out.tri_off.resize(n + 1);
    out.edge_off.resize(n + 1);
    std::vector<int32_t> goff(n + 1);
    int32_t S = 0, E = 0, T = 0, G = 0;
    for (int32_t i = 0; i < n; i++) {
        const uint32_t s = mu::measure(m, i);
        out.cell_ptr[i] = S;
        out.edge_off[i] = E;
        out.tri_off[i] = T;
        goff[i] = G;
        S += s & 255;
        E += s >> 8 & 255;
        T += s >> 16 & 255;
        G += s >> 24;
    }
    out.cell_ptr[n] = S;
    out.edge_off[n] = E;
    out.tri_off[n] = T;
    out.n_edges = E;
    out.n_tris = T;
    out.g = G;
    out.slot_nb.resize(S);
    out.gx.resize(G); out.gy.resize(G); out.ghost_src.resize(G); out.ghost_xf.resize(G);
    out.ghost_shift.resize(G); out.ghost_img.resize(G);
    m.out_ptr = out.cell_ptr.data();
    m.out_nb = out.slot_nb.data();
    m.tri_off = out.tri_off.data();
    m.edge_off = out.edge_off.data();
    m.ghost_off = goff.data();
    m.gx = out.gx.data(); m.gy = out.gy.data(); m.gsrc = out.ghost_src.data(); m.gxf = out.ghost_xf.data();
    m.gshift = out.ghost_shift.data(); m.gimg = out.ghost_img.data();
    for (int32_t i = 0; i < n; i++) mu::place_ghosts(m, i);
    for (int32_t i = 0; i < n; i++) mu::place_ring(m, i);
    if (flags) return 0;
    out.band = ip.band;
    out.cell_order.resize(n);
    degree_order(n, out.cell_ptr.data(), out.cell_order.data());
    mesh = std::move(out);
    return 1;
}

}  // namespace rich
