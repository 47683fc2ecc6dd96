// rich_proxy.cpp -- host builder of the surface proxies (rich_proxy.h).
//
// Each surface's triangles (the triangles that share a BVH surface subtree)
// are fitted by a plane or, by linear least squares on |v|^2 = 2 c . v + k, by
// a sphere; surfaces that follow the same one are merged, so that the tiles of
// one mirror cost a ray one crossing. Everything that the ray side relies on
// (shell thickness, grid lists) is measured from the FP32 values that the
// kernel reads.
#include "rich_proxy.h"

#include "rich_bvh.h"

#include <algorithm>
#include <array>
#include <cstring>
#include <map>

namespace rich {

namespace {

using V3 = std::array<double, 3>;

constexpr double kUnit = 1.0 / 16777216.0;   // 2^-24
constexpr int32_t kNoSurf32 = 0x7FFFFFFF;
// Cells of kCellScale of the root mean triangle area, at least four margins wide; at
// most kMaxCellsPerTri cells a triangle and 4096 in a mesh, and kMaxCells in all (96 MB,
// which the L2 holds). 0.12 of the area is 70 cells a triangle, more where the mesh fills
// less than its bounding rectangle, so above some 700 triangles the number of cells
// is what the limit a triangle leaves: 1.43e6 cells on RICH1 (65 a triangle, 11.4 MB),
// 9.57e6 on RICH2 (64, 76.5 MB); most list one triangle. Trace of RICH1, 10^4 tracks,
// with 16, 31 and 65 cells a triangle (0.25 and 0.18 of the area, and the limit): 458,
// 442, 428 us; of RICH2, 1.2 x 10^5 tracks, with 18, 35 and 64: 3.54, 3.42, 3.34 ms (and
// 835 us, 7.33 ms with one, before later steps). More than 65 were not measured.
constexpr double kCellScale = 0.12;
constexpr double kMaxCellsPerTri = 64.0;
constexpr double kMaxCells = 1.2e7;

V3 vert(const DevTri &t, int k) {
    return k == 0 ? V3{t.v0x, t.v0y, t.v0z}
                  : (k == 1 ? V3{t.v1x, t.v1y, t.v1z} : V3{t.v2x, t.v2y, t.v2z});
}
V3 sub(const V3 &a, const V3 &b) { return {a[0] - b[0], a[1] - b[1], a[2] - b[2]}; }
double dot(const V3 &a, const V3 &b) { return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]; }
V3 cross(const V3 &a, const V3 &b) {
    return {a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]};
}
double len(const V3 &a) { return std::sqrt(dot(a, a)); }
V3 tri_cross(const DevTri &t) {
    const V3 a = vert(t, 0);
    return cross(sub(vert(t, 1), a), sub(vert(t, 2), a));
}

// A sphere (r > 0) or plane (r = 0, unit normal n) with FP32 values, and the
// triangles on it.
struct Fit {
    V3 c{}, n{};
    double r = 0.0;
    double shell = 0.0;       // largest distance of a point of a facet from it
    std::vector<int> tris;
};

// Largest |o| of an origin in the scene's box [-extent, extent]^3.
double o_max(double extent) { return 1.75 * extent; }

V3 round32(const V3 &a) { return {(double)(float)a[0], (double)(float)a[1], (double)(float)a[2]}; }

// Largest distance of the triangles from the sphere or plane: for a sphere
// between the farthest vertex and the nearest point of the facet's plane.
double shell_of(const Fit &f, const std::vector<DevTri> &T, const std::vector<int> &sel,
                size_t stride = 1) {
    double s = 0.0;
    for (size_t at = 0; at < sel.size(); at += stride) {
        const int i = sel[at];
        V3 w[3];
        for (int k = 0; k < 3; ++k) w[k] = sub(vert(T[i], k), f.c);
        if (f.r > 0.0) {
            const V3 g = tri_cross(T[i]);
            const double gl = len(g);
            double lo = gl > 0.0 ? std::fabs(dot(w[0], g)) / gl : 0.0;
            for (int k = 0; k < 3; ++k) {
                s = std::max(s, std::fabs(len(w[k]) - f.r));
                if (!(gl > 0.0)) lo = std::max(lo, len(w[k]));   // degenerate: its vertices
            }
            s = std::max(s, std::fabs(f.r - lo));
        } else {
            for (int k = 0; k < 3; ++k) s = std::max(s, std::fabs(dot(w[k], f.n)));
        }
    }
    return s;
}

bool fit_plane(const std::vector<DevTri> &T, const std::vector<int> &sel, Fit &f) {
    V3 n{}, c{};
    for (int i : sel) {
        V3 g = tri_cross(T[i]);
        if (dot(g, n) < 0.0) g = {-g[0], -g[1], -g[2]};   // either winding
        for (int k = 0; k < 3; ++k) {
            n[k] += g[k];
            for (int v = 0; v < 3; ++v) c[k] += vert(T[i], v)[k];
        }
    }
    const double l = len(n);
    if (!(l > 0.0)) return false;
    for (int k = 0; k < 3; ++k) {
        n[k] /= l;
        c[k] /= 3.0 * (double)sel.size();
    }
    f.c = round32(c);
    f.n = round32(n);
    f.r = 0.0;
    f.shell = shell_of(f, T, sel);
    return true;
}

bool fit_sphere(const std::vector<DevTri> &T, const std::vector<int> &sel, Fit &f) {
    V3 m{};
    for (int i : sel)
        for (int v = 0; v < 3; ++v)
            for (int k = 0; k < 3; ++k) m[k] += vert(T[i], v)[k] / (3.0 * (double)sel.size());
    double scale = 0.0;
    for (int i : sel)
        for (int v = 0; v < 3; ++v) scale = std::max(scale, len(sub(vert(T[i], v), m)));
    if (!(scale > 0.0)) return false;
    // normal equations of |p|^2 = a . p + k, p = (v - m) / scale
    double A[4][5] = {};
    for (int i : sel)
        for (int v = 0; v < 3; ++v) {
            const V3 p = sub(vert(T[i], v), m);
            const double row[5] = {p[0] / scale, p[1] / scale, p[2] / scale, 1.0,
                                   dot(p, p) / (scale * scale)};
            for (int a = 0; a < 4; ++a)
                for (int b = 0; b < 5; ++b) A[a][b] += row[a] * row[b];
        }
    for (int a = 0; a < 4; ++a) {
        int piv = a;
        for (int b = a + 1; b < 4; ++b)
            if (std::fabs(A[b][a]) > std::fabs(A[piv][a])) piv = b;
        if (!(std::fabs(A[piv][a]) > 1e-14 * A[3][3])) return false;
        std::swap(A[a], A[piv]);
        for (int b = 0; b < 4; ++b) {
            if (b == a) continue;
            const double q = A[b][a] / A[a][a];
            for (int k = a; k < 5; ++k) A[b][k] -= q * A[a][k];
        }
    }
    double x[4];
    for (int a = 0; a < 4; ++a) x[a] = A[a][4] / A[a][a];
    f.c = round32({m[0] + 0.5 * x[0] * scale, m[1] + 0.5 * x[1] * scale, m[2] + 0.5 * x[2] * scale});
    // radius in the middle of the facets' distances
    double lo = HUGE_VAL, hi = 0.0;
    for (int i : sel) {
        const V3 g = tri_cross(T[i]);
        const double gl = len(g);
        if (gl > 0.0) lo = std::min(lo, std::fabs(dot(sub(vert(T[i], 0), f.c), g)) / gl);
        for (int v = 0; v < 3; ++v) hi = std::max(hi, len(sub(vert(T[i], v), f.c)));
    }
    if (!std::isfinite(lo) || !std::isfinite(hi)) return false;
    f.r = (double)(float)(0.5 * (lo + hi));
    f.n = {};
    f.shell = shell_of(f, T, sel);
    return f.r > 0.0;
}

// Longest way along a ray from its crossing of the sphere or plane, at a cosine of
// at least kProxyCosMin, to a point within the shell (and the rounding error E). To
// a plane's it is depth / cosine. Inside a sphere the ray flattens on its way: from
// radius r at cosine c to radius r - s it is r c - sqrt(r^2 c^2 - 2 r s + s^2), longer
// than s / c by some s^2 (1 - c^2) / (2 r c^3) (outwards it is shorter than s / c). 0:
// a ray at the limit does not come as deep as s, and no such bound holds. The squared
// cosine of a crossing that passes the FP32 test may be below the limit by E / r
// (16 u W / r from q2 and 4 u from r^2, W >= r).
double shell_reach(const Fit &f, double E) {
    const double s = f.shell + E;
    if (!(f.r > 0.0)) return s / kProxyCosMin;
    const double c2 = (double)kProxyCosMin * kProxyCosMin - E / f.r;
    const double in2 = f.r * f.r * c2 - 2.0 * f.r * s + s * s;
    if (!(c2 > 0.0 && in2 > 0.0 && s < f.r)) return 0.0;
    return f.r * std::sqrt(c2) - std::sqrt(in2);
}

// Grid and device record of one fit; false when the margin does not suit it.
bool make_proxy(const std::vector<DevTri> &T, const Fit &f, double extent, ProxyResult &out) {
    const bool sphere = f.r > 0.0;
    // axis and grid axes (FP32; only their linear map matters below)
    V3 axis = f.n;
    if (sphere) {
        axis = {};
        for (int i : f.tris)
            for (int v = 0; v < 3; ++v) {
                const V3 w = sub(vert(T[i], v), f.c);
                const double l = len(w);
                for (int k = 0; k < 3; ++k) axis[k] += w[k] / l;
            }
        const double l = len(axis);
        if (!(l > 0.0)) return false;
        for (double &a : axis) a /= l;
        axis = round32(axis);
    }
    const V3 h = std::fabs(axis[0]) < 0.6 ? V3{1.0, 0.0, 0.0} : V3{0.0, 1.0, 0.0};
    V3 e1 = cross(h, axis);
    const double l1 = len(e1);
    for (double &a : e1) a /= l1;
    const V3 e2 = round32(cross(axis, e1));
    e1 = round32(e1);
    double lo[3], hi[3], area = 0.0;
    for (int k = 0; k < 3; ++k) {
        lo[k] = HUGE_VAL;
        hi[k] = -HUGE_VAL;
    }
    for (int i : f.tris) {
        area += 0.5 * len(tri_cross(T[i]));
        for (int v = 0; v < 3; ++v) {
            const V3 w = sub(vert(T[i], v), f.c);
            const double q[3] = {dot(w, e1), dot(w, e2), dot(w, axis)};
            for (int k = 0; k < 3; ++k) {
                lo[k] = std::min(lo[k], q[k]);
                hi[k] = std::max(hi[k], q[k]);
            }
        }
    }
    // the projection along the axis stays well away from the sphere's rim
    if (sphere && !(lo[2] >= 0.5 * f.r)) return false;
    // sphere bounding the mesh, about the box's centre
    V3 g{};
    for (int k = 0; k < 3; ++k)
        g[k] = f.c[k] + 0.5 * (lo[0] + hi[0]) * e1[k] + 0.5 * (lo[1] + hi[1]) * e2[k] +
               0.5 * (lo[2] + hi[2]) * axis[k];
    g = round32(g);
    double rho = 0.0;
    for (int i : f.tris)
        for (int v = 0; v < 3; ++v) rho = std::max(rho, len(sub(vert(T[i], v), g)));
    // distances from c up to which the bounds are to hold (origins anywhere in
    // the scene's box), and the margins
    const double W = o_max(extent) + len(f.c), W_g = o_max(extent) + len(g);
    const double E = 32.0 * kUnit * W;
    const double reach = shell_reach(f, E);
    if (!(reach > 0.0)) return false;
    const double margin = reach + E;
    const double tri_size = std::sqrt(area / (double)f.tris.size());
    double size = std::max(kCellScale * tri_size, 4.0 * margin);
    const double wx = hi[0] - lo[0] + 4.0 * margin, wy = hi[1] - lo[1] + 4.0 * margin;
    const double share = (double)f.tris.size() / (double)T.size();
    const double most = std::min(kMaxCellsPerTri * (double)f.tris.size(), kMaxCells * share) + 4096.0;
    if (wx * wy > most * size * size) size = std::sqrt(wx * wy / most);
    // long thin meshes: no more than `most` cells along either side
    size = std::max(size, std::max(wx, wy) / most);
    if (!(size > 0.0) || !(4.0 * margin <= tri_size)) return false;
    // cell coordinates: FP32 axes divided by the cell size (only their linear
    // map matters) and FP32 corner
    const V3 f1 = round32({e1[0] / size, e1[1] / size, e1[2] / size});
    const V3 f2 = round32({e2[0] / size, e2[1] / size, e2[2] / size});
    const double m = margin / size * (1.0 + 1.0e-6);
    const float x0 = (float)(lo[0] / size - 2.0 * m), y0 = (float)(lo[1] / size - 2.0 * m);
    const int nx = (int)std::ceil(hi[0] / size + 2.0 * m - x0) + 1;
    const int ny = (int)std::ceil(hi[1] / size + 2.0 * m - y0) + 1;
    if ((double)nx * ny > 2.0e8) return false;
    DevProxy P;
    std::memset(&P, 0, sizeof P);
    P.cx = (float)f.c[0]; P.cy = (float)f.c[1]; P.cz = (float)f.c[2]; P.r = (float)f.r;
    P.dt = (float)margin;
    P.ax = (float)axis[0]; P.ay = (float)axis[1]; P.az = (float)axis[2];
    P.z_min = (float)std::min(0.5 * lo[2], lo[2] - margin);
    P.e1x = (float)f1[0]; P.e1y = (float)f1[1]; P.e1z = (float)f1[2]; P.x0 = x0;
    P.e2x = (float)f2[0]; P.e2y = (float)f2[1]; P.e2z = (float)f2[2]; P.y0 = y0;
    P.fnx = (float)nx; P.fny = (float)ny; P.nx = nx;
    P.r2 = (float)(f.r * f.r);
    P.h2_min = (float)(f.r * f.r * kProxyCosMin * kProxyCosMin);
    const double out_r = f.r + f.shell + 2.0 * E + 4.0e-6 * W;
    P.q2_max = (float)(out_r * out_r);
    // a direction that is unit to 1e-6 puts the first estimate off by at most
    // 1e-6 t^2 / h, t <= 2 W and h >= r cos_min
    P.t_far = (float)(-(double)P.dt - (sphere ? 4.0e-6 * W * W / (f.r * kProxyCosMin) : 0.0));
    P.gx = (float)g[0]; P.gy = (float)g[1]; P.gz = (float)g[2];
    const double g_r = rho + E + P.dt + 4.0e-6 * W_g;
    P.g_r = (float)(g_r * (1.0 + 1.0e-6));
    // (a direction that is unit to 1e-6 changes (w . d)^2 by 2e-6 W^2 at most)
    P.g2 = (float)((g_r * g_r + (16.0 * kUnit + 2.0e-6) * W_g * W_g) * (1.0 + 1.0e-6));
    // the triangles whose projection comes within the margin of each cell (the
    // triangle's edges and the widened cell, by separating axes), row by row
    // the first two triangles of a cell go into it, further ones aside
    std::vector<DevProxyCell> &cells = out.cells[0];
    cells.assign((size_t)nx * ny, DevProxyCell{-1, -1});
    std::vector<std::pair<int32_t, int32_t>> more;        // (cell, triangle)
    // one surface, or several apart: a photon that leaves a facet starts within
    // the margin of it, so the cell of its start lists that facet's surface
    bool single = true, apart = true;
    for (int i : f.tris) {
        single = single && T[i].pad == T[f.tris[0]].pad;
        apart = apart && T[i].pad != kNoSurf32;
    }
    for (int i : f.tris) {
        double q[3][2], blo[2] = {HUGE_VAL, HUGE_VAL}, bhi[2] = {-HUGE_VAL, -HUGE_VAL};
        for (int v = 0; v < 3; ++v) {
            const V3 w = sub(vert(T[i], v), f.c);
            q[v][0] = dot(w, f1) - (double)x0;
            q[v][1] = dot(w, f2) - (double)y0;
            for (int k = 0; k < 2; ++k) {
                blo[k] = std::min(blo[k], q[v][k] - m);
                bhi[k] = std::max(bhi[k], q[v][k] + m);
            }
        }
        const double turn = (q[1][0] - q[0][0]) * (q[2][1] - q[0][1]) -
                            (q[1][1] - q[0][1]) * (q[2][0] - q[0][0]);
        const double sg = turn < 0.0 ? -1.0 : 1.0;
        const int iy0 = std::max(0, (int)std::floor(blo[1]));
        const int iy1 = std::min(ny - 1, (int)std::floor(bhi[1]));
        const double half = 0.5 + m;
        // outward normal of each edge and the bound of its half plane, widened
        // by the cell
        double ex[3], ey[3], rhs[3];
        for (int v = 0; v < 3; ++v) {
            const double *a = q[v], *b = q[(v + 1) % 3];
            ex[v] = sg * (b[1] - a[1]);
            ey[v] = -sg * (b[0] - a[0]);
            rhs[v] = (std::fabs(ex[v]) + std::fabs(ey[v])) * half * (1.0 + 1.0e-9) + ex[v] * a[0] +
                     ey[v] * a[1];
        }
        for (int iy = iy0; iy <= iy1; ++iy) {
            // the cells of a row that meet the triangle are consecutive
            const double my = iy + 0.5;
            double lo_x = blo[0] - 0.5, hi_x = bhi[0] + 0.5;       // of the cell's centre
            for (int v = 0; v < 3; ++v) {
                const double r = rhs[v] - ey[v] * my;
                if (ex[v] > 0.0)
                    hi_x = std::min(hi_x, r / ex[v]);
                else if (ex[v] < 0.0)
                    lo_x = std::max(lo_x, r / ex[v]);
                else if (r < 0.0)
                    hi_x = -1.0;
            }
            const int ix0 = std::max(0, (int)std::ceil(lo_x - 0.5 - 1.0e-6));
            const int ix1 = std::min(nx - 1, (int)std::floor(hi_x - 0.5 + 1.0e-6));
            DevProxyCell *row = cells.data() + (size_t)iy * nx;
            for (int ix = ix0; ix <= ix1; ++ix) {
                DevProxyCell &d = row[ix];
                if (d.a < 0) {
                    d.a = i;
                    continue;
                }
                apart = apart && T[d.a].pad == T[i].pad;
                if (d.b < 0)
                    d.b = i;
                else
                    more.push_back({iy * nx + ix, i});
            }
        }
    }
    std::sort(more.begin(), more.end());
    for (size_t k = 0; k < more.size();) {
        DevProxyCell &d = cells[(size_t)more[k].first];
        const size_t first = out.lists.size();
        out.lists.push_back(d.a);
        out.lists.push_back(d.b);
        out.list_cells.push_back(more[k].first);
        const int32_t cell = more[k].first;
        for (; k < more.size() && more[k].first == cell; ++k) out.lists.push_back(more[k].second);
        d.a = (int32_t)first;
        d.b = (int32_t)(0x80000000u | (uint32_t)(out.lists.size() - first));
    }
    if (T[f.tris[0]].pad != kNoSurf32)
        P.code = single ? (int32_t)kProxySingle : (apart ? (int32_t)kProxyApart : 0);
    out.proxies.push_back(P);
    return true;
}

}  // namespace

void build_proxies(const std::vector<DevTri> &T, double extent, ProxyResult &out) {
    out = ProxyResult();
    if (T.empty()) return;
    std::map<int32_t, std::vector<int>> groups;
    for (size_t i = 0; i < T.size(); ++i) groups[T[i].pad].push_back((int)i);
    std::vector<const std::vector<int> *> order;
    for (auto &[ref, sel] : groups) order.push_back(&sel);
    std::stable_sort(order.begin(), order.end(),
                     [](const auto *a, const auto *b) { return a->size() > b->size(); });
    // what FP32 vertices of a plane or sphere may be off it
    const double tol = 8.0 * kUnit * extent;
    // each surface by itself, then merged in order
    struct Own {
        Fit f;
        bool flat, ok;
    };
    std::vector<Own> own(order.size());
    run_parallel(order.size(), [&](size_t i) {
        Own &o = own[i];
        o.flat = fit_plane(T, *order[i], o.f) && o.f.shell <= tol;
        o.ok = o.flat || fit_sphere(T, *order[i], o.f);
    });
    std::vector<Fit> fits;
    for (size_t i = 0; i < order.size(); ++i) {
        const Own &o = own[i];
        if (!o.ok) return;
        Fit *home = nullptr;
        for (Fit &f : fits) {
            if ((f.r > 0.0) == o.flat) continue;
            // (a sample decides; the merged fit below is measured in full)
            if (shell_of(f, T, *order[i], order[i]->size() / 64 + 1) <=
                2.0 * (o.flat ? 0.0 : o.f.shell) + 4.0 * tol) {
                home = &f;
                break;
            }
        }
        if (!home) {
            if (fits.size() == RICH_MAX_PROXIES) return;
            fits.push_back(o.f);
            home = &fits.back();
        }
        home->tris.insert(home->tris.end(), order[i]->begin(), order[i]->end());
    }
    std::stable_sort(fits.begin(), fits.end(),
                     [](const Fit &a, const Fit &b) { return a.r == 0.0 && b.r > 0.0; });
    // all surfaces of a fit together, then its grid
    std::vector<ProxyResult> part(fits.size());
    run_parallel(fits.size(), [&](size_t k) {
        Fit &f = fits[k];
        part[k].cells.resize(1);
        const bool ok = f.r > 0.0 ? fit_sphere(T, f.tris, f) : fit_plane(T, f.tris, f);
        if (!ok || !make_proxy(T, f, extent, part[k])) part[k] = ProxyResult();
    });
    out.tri_code.assign(T.size(), 0u);
    size_t n_cells = 0;
    for (ProxyResult &p : part) {
        if (p.proxies.empty() || n_cells + p.cells[0].size() > (size_t)2e8) {
            out = ProxyResult();
            return;
        }
        for (int i : fits[out.proxies.size()].tris)
            out.tri_code[i] = (uint32_t)p.proxies[0].code | (uint32_t)(out.proxies.size() + 1);
        out.proxies.push_back(p.proxies[0]);
        out.proxies.back().first_cell = (int32_t)n_cells;
        for (int32_t cell : p.list_cells) p.cells[0][(size_t)cell].a += (int32_t)out.lists.size();
        out.lists.insert(out.lists.end(), p.lists.begin(), p.lists.end());
        n_cells += p.cells[0].size();
        out.cells.push_back(std::move(p.cells[0]));
        out.n_planes += p.proxies[0].r == 0.0f;
        out.dt_max = std::max(out.dt_max, p.proxies[0].dt);
    }
    out.o2_max = (float)(o_max(extent) * o_max(extent));
}

}  // namespace rich
