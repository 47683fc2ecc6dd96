"""Surface proxies of meshed mirrors (rich_proxy), on the CPU: the ray side
compiled for the host beside the builder.

The property the trace relies on: a ray that meets a triangle is either left
to the BVH or finds that triangle in the cell of one of its crossings. Rays
are aimed at points of every kind of triangle, edges and corners included,
with FP32 origins and directions; grazing and distant ones too. Rays that have
just left a facet pass over its surface and still find the next one."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2309_12496_gb300 import build
from paper_2309_12496_gb300 import workloads as W

WRAP = r"""
#include "rich_bvh.h"
#include "rich_proxy.h"
#include <algorithm>
#include <cstring>
using namespace rich;
extern "C" int proxy_find(int64_t nt, const float *v, const int32_t *surf, double extent, int64_t nr,
                          const float *o, const float *d, const int32_t *target, float t_max,
                          uint8_t *out, double *listed, const double *t_hit, double *reach) {
    BvhResult b;
    std::string err;
    if (!build_bvh(v, surf, nt, b, err)) return -1;
    std::vector<DevTri> T((size_t)nt);
    std::vector<int> pos((size_t)nt);
    for (int64_t k = 0; k < nt; ++k) {
        const int s = b.leaf_order[(size_t)k];
        std::memset(&T[(size_t)k], 0, sizeof(DevTri));
        std::memcpy(&T[(size_t)k], v + 9 * (int64_t)s, 36);
        T[(size_t)k].pad = b.surface_ref[(size_t)k];
        pos[(size_t)s] = (int)k;
    }
    ProxyResult R;
    build_proxies(T, extent, R);
    double tests = 0;
    for (int64_t i = 0; i < nr; ++i) {
        out[i] = 0;
        const float *O = o + 3 * i, *D = d + 3 * i;
        if (!(O[0] * O[0] + O[1] * O[1] + O[2] * O[2] <= R.o2_max)) {
            out[i] = 2;
            continue;
        }
        for (size_t k = 0; k < R.proxies.size(); ++k) {
            const DevProxy &P = R.proxies[k];
            int cell[2] = {-1, -1};
            float t, t_in = 0.0f, b2, h2;
            bool sure, entering = false;
            if (proxy_misses(P, O[0], O[1], O[2], D[0], D[1], D[2], t_max)) continue;
            if ((int)k < R.n_planes) {
                cell[0] = proxy_plane(P, O[0], O[1], O[2], D[0], D[1], D[2], 1e-3f, t_max, t, sure);
            } else {
                cell[0] = proxy_sphere(P, O[0], O[1], O[2], D[0], D[1], D[2], 1e-3f, t_max, t, sure,
                                       entering, b2, h2);
                if (entering)
                    cell[1] = proxy_sphere_side(P, O[0] - P.cx, O[1] - P.cy, O[2] - P.cz, D[0], D[1],
                                                D[2], b2, h2, -1.0f, 1e-3f, t_max, t_in, true);
            }
            if (!sure) out[i] |= 2;
            if (t_hit && sure) {
                double far = std::fabs(t - t_hit[i]);
                if (entering) far = std::min(far, std::fabs(t_in - t_hit[i]));
                *reach = std::max(*reach, far / P.dt);
            }
            for (int c : cell) {
                if (c < 0) continue;
                const DevProxyCell &L = R.cells[k][(size_t)(c - P.first_cell)];
                const bool list = L.b < -1;
                const int n = list ? (L.b & 0x7FFFFFFF) : (L.a >= 0) + (L.b >= 0);
                tests += n;
                for (int q = 0; q < n; ++q)
                    if ((list ? R.lists[(size_t)L.a + q] : (q ? L.b : L.a)) == pos[target[i]]) out[i] |= 1;
            }
        }
    }
    *listed = nr ? tests / (double)nr : 0.0;
    return (int)R.proxies.size();
}
struct HostProxies {
    const std::vector<DevProxy> *v;
    int n_proxies;
    const DevProxy *proxies() const { return v->data(); }
};
// The cells that the trace looks up for rays that have just left triangle
// from[i]: out 1 when target[i], met at t_hit[i], is listed there (or -1, none), 2 when
// the ray goes to the BVH. used: proxy codes of the triangles, and the number of rays
// for which the code passed over a crossing.
extern "C" int proxy_leave(int64_t nt, const float *v, const int32_t *surf, double extent, int64_t nr,
                           const float *o, const float *d, const int32_t *from,
                           const int32_t *target, const double *t_hit, uint8_t *out,
                           uint32_t *codes, int64_t *used) {
    BvhResult b;
    std::string err;
    if (!build_bvh(v, surf, nt, b, err)) return -1;
    std::vector<DevTri> T((size_t)nt);
    std::vector<int> pos((size_t)nt);
    for (int64_t k = 0; k < nt; ++k) {
        const int s = b.leaf_order[(size_t)k];
        std::memset(&T[(size_t)k], 0, sizeof(DevTri));
        std::memcpy(&T[(size_t)k], v + 9 * (int64_t)s, 36);
        T[(size_t)k].pad = b.surface_ref[(size_t)k];
        pos[(size_t)s] = (int)k;
    }
    ProxyResult R;
    build_proxies(T, extent, R);
    if (R.proxies.empty()) return 0;
    std::vector<DevProxyCell> cells;
    for (auto &grid : R.cells) cells.insert(cells.end(), grid.begin(), grid.end());
    for (int64_t k = 0; k < nt; ++k) codes[k] = R.tri_code[(size_t)pos[(size_t)k]];
    const HostProxies S{&R.proxies, (int)R.proxies.size()};
    auto lists = [&](int c, int tri) {
        if (c < 0) return false;
        const DevProxyCell &L = cells[(size_t)c];
        if (L.b >= -1) return L.a == tri || L.b == tri;
        for (int q = 0; q < (L.b & 0x7FFFFFFF); ++q)
            if (R.lists[(size_t)L.a + q] == tri) return true;
        return false;
    };
    *used = 0;
    for (int64_t i = 0; i < nr; ++i) {
        const float *O = o + 3 * i, *D = d + 3 * i;
        const uint32_t code = codes[from[i]];
        const ProxyCells q = proxy_cells(S, R.n_planes, O[0], O[1], O[2], D[0], D[1], D[2], code,
                                         1e-3f, 3e38f);
        const ProxyCells q0 = proxy_cells(S, R.n_planes, O[0], O[1], O[2], D[0], D[1], D[2], 0u,
                                          1e-3f, 3e38f);
        *used += q.c0 != q0.c0 || q.c1 != q0.c1 || q.t2 != q0.t2 || q.sure != q0.sure;
        const double t = target[i] < 0 ? 3e38 : t_hit[i];
        const bool second = q.c1 >= 0 && q.t1 <= t + R.dt_max;
        out[i] = 0;
        if (!q.sure || (q.c0 >= 0 && !(q.t2 > t + R.dt_max))) out[i] |= 2;
        const int tri = target[i] < 0 ? -1 : pos[(size_t)target[i]];
        if (tri < 0 || lists(q.c0, tri) || (second && lists(q.c1, tri))) out[i] |= 1;
    }
    return S.n_proxies;
}
// The nearest triangle ahead of each ray in FP64 that is not of the surface of
// triangle from[i] (from may be null); -1: none; -2: met within 1e-3 of an edge (where
// FP32 may see its neighbour).
extern "C" void nearest_tri(int64_t nt, const float *v, const int32_t *surf, int64_t nr,
                            const float *o, const float *d, const int32_t *from, int32_t *target,
                            double *t_hit) {
    for (int64_t i = 0; i < nr; ++i) {
        const double O[3] = {o[3 * i], o[3 * i + 1], o[3 * i + 2]};
        const double D[3] = {d[3 * i], d[3 * i + 1], d[3 * i + 2]};
        double best = 1e300;
        target[i] = -1;
        for (int64_t k = 0; k < nt; ++k) {
            if (from && (k == from[i] || (surf && surf[k] == surf[from[i]]))) continue;
            double a[3], e1[3], e2[3];
            for (int c = 0; c < 3; ++c) {
                a[c] = O[c] - v[9 * k + c];
                e1[c] = (double)v[9 * k + 3 + c] - v[9 * k + c];
                e2[c] = (double)v[9 * k + 6 + c] - v[9 * k + c];
            }
            const double p[3] = {D[1] * e2[2] - D[2] * e2[1], D[2] * e2[0] - D[0] * e2[2],
                                 D[0] * e2[1] - D[1] * e2[0]};
            const double q[3] = {a[1] * e1[2] - a[2] * e1[1], a[2] * e1[0] - a[0] * e1[2],
                                 a[0] * e1[1] - a[1] * e1[0]};
            const double det = e1[0] * p[0] + e1[1] * p[1] + e1[2] * p[2];
            if (det == 0.0) continue;
            const double b1 = (a[0] * p[0] + a[1] * p[1] + a[2] * p[2]) / det;
            const double b2 = (D[0] * q[0] + D[1] * q[1] + D[2] * q[2]) / det;
            const double t = (e2[0] * q[0] + e2[1] * q[1] + e2[2] * q[2]) / det;
            const double in = std::min(std::min(b1, b2), 1.0 - b1 - b2);
            if (in < -1e-3 || t < 1e-2 || t >= best) continue;
            best = t;
            t_hit[i] = t;
            target[i] = in >= 1e-3 ? (int32_t)k : -2;
        }
    }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("proxy")
    src, so = d / "wrap.cpp", d / "wrap.so"
    src.write_text(WRAP)
    cuda = os.path.join(os.path.dirname(os.path.dirname(shutil.which("nvcc") or
                                                        "/usr/local/cuda/bin/nvcc")), "include")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off", "-I", cuda,
                    "-I", build.INCLUDE, "-I", build.CSRC, str(src),
                    os.path.join(build.CSRC, "rich_bvh.cpp"),
                    os.path.join(build.CSRC, "rich_proxy.cpp"), "-o", str(so)], check=True)
    return C.CDLL(str(so))


def _patch(radius, half, cells, axis_turn, shift=0.0):
    """One smooth square patch of a sphere (or a plane, radius 0), turned and
    moved by arbitrary amounts."""
    rng = np.random.default_rng(int(radius + cells))
    q, _ = np.linalg.qr(rng.standard_normal((3, 3)) * axis_turn + np.eye(3))
    at = rng.uniform(-1, 1, 3) * shift
    if radius:
        tris, _ = W._mesh_rect_tile(at, radius, q[2], q[0], q[1], -half, half, -half, half, cells,
                                    cells)
    else:
        tris = W._mesh_rectangle(at, q[0], q[1], 2 * half, 1.3 * half, cells, cells)
    return tris.astype(np.float32), np.zeros(len(tris), np.int32)


SCENES = {
    "rich1": lambda: (W.rich1_scene().tri_vertices, W.rich1_scene().tri_surface),
    "rich2": lambda: (W.rich2_scene(hex_subdiv=6).tri_vertices,
                      W.rich2_scene(hex_subdiv=6).tri_surface),
    "point": lambda: (W.point_source_scene(meshed=True).tri_vertices, None),
    "sphere_small": lambda: _patch(500.0, 200.0, 9, 1.0, 300.0),
    "plane_turned": lambda: _patch(0.0, 350.0, 7, 2.0, 2000.0),
    "plane_two_triangles": lambda: _patch(0.0, 100.0, 1, 1.0, 10.0),
}


def _find(lib, v, surf, extent, o, d, k, t_hit=None):
    """proxy_find on rays (o, d) with target triangles k, met at t_hit: proxies,
    flags, and the largest distance along a ray from its crossing to the
    triangle, as a share of the bound (one proxy)."""
    out = np.zeros(len(o), np.uint8)
    listed, reach = C.c_double(), C.c_double()
    p = [None if a is None else a.ctypes.data_as(C.c_void_p)
         for a in (v, None if surf is None else np.ascontiguousarray(surf, np.int32),
                   o, d, k, out, t_hit)]
    n = lib.proxy_find(C.c_int64(len(v)), p[0], p[1], C.c_double(extent), C.c_int64(len(o)), p[2],
                       p[3], p[4], C.c_float(3e38), p[5], C.byref(listed), p[6], C.byref(reach))
    return n, out, reach.value


def _rays(v, n, rng, cos_min, dist):
    """Rays at points of random triangles: inside, on edges, at corners."""
    k = rng.integers(0, len(v), n)
    b = rng.dirichlet((0.6, 0.6, 0.6), n)
    kind = rng.integers(0, 4, n)
    b[kind == 1, 0] = 0.0
    b[kind == 2] = np.eye(3)[rng.integers(0, 3, int((kind == 2).sum()))]
    b /= b.sum(1, keepdims=True)
    t = v[k].astype(np.float64)
    p = np.einsum("ij,ijk->ik", b, t)
    nrm = np.cross(t[:, 1] - t[:, 0], t[:, 2] - t[:, 0])
    nrm /= np.linalg.norm(nrm, axis=1, keepdims=True)
    c = rng.uniform(cos_min, 1.0, n) * rng.choice([-1.0, 1.0], n)
    side = rng.standard_normal((n, 3))
    side -= (side * nrm).sum(1, keepdims=True) * nrm
    side /= np.linalg.norm(side, axis=1, keepdims=True)
    d = c[:, None] * nrm + np.sqrt(1 - c * c)[:, None] * side
    o = p - d * np.exp(rng.uniform(np.log(1.0), np.log(dist), n))[:, None]
    return k.astype(np.int32), o.astype(np.float32), d.astype(np.float32)


@pytest.mark.parametrize("name", sorted(SCENES))
@pytest.mark.parametrize("cos_min,dist", [(0.3, 4000.0), (0.0, 4000.0), (0.3, 60000.0)])
def test_a_ray_finds_the_triangle_it_meets_or_goes_to_the_bvh(lib, name, cos_min, dist):
    v, surf = SCENES[name]()
    v = np.ascontiguousarray(v, np.float32)
    n = 60000
    k, o, d = _rays(v, n, np.random.default_rng(len(v)), cos_min, dist)
    n_proxies, out, _ = _find(lib, v, surf, float(np.abs(v).max()), o, d, k)
    assert n_proxies == {"rich1": 4, "rich2": 5}.get(name, 1)
    assert np.all(out != 0), (int((out == 0).sum()), np.flatnonzero(out == 0)[:5])
    if cos_min > 0.25 and dist < 5000:
        assert (out & 1).mean() > 0.5            # most by their cells


# (radius, half width, cells): facet edges of 0.1 to 0.4 of the radius, the
# builder's limit among them, and whether they get a proxy
COARSE = {"r500_10": (500.0, 100.0, 4, 1), "r2700_18": (2700.0, 500.0, 2, 1),
          "r500_20": (500.0, 150.0, 3, 1), "r1000_25": (1000.0, 250.0, 2, 1),
          "r500_27": (500.0, 200.0, 3, 1), "r500_30": (500.0, 150.0, 2, 1),
          "r1000_30": (1000.0, 300.0, 2, 1), "r2700_30": (2700.0, 800.0, 2, 1),
          "r500_40": (500.0, 200.0, 2, 0)}


@pytest.mark.parametrize("name", sorted(COARSE))
def test_coarse_facets_are_found_at_the_steepest_crossings(lib, name):
    """The shell between a sphere and its facets is thick here against the
    radius, and a ray near the cosine limit runs through it for longer than its
    thickness over the cosine. Rays at the deepest points of the facets
    (the middles of edges, a little inside) that cross the proxy's sphere at
    cosines 0.24 to 0.3, checked on the triangle that they meet first and on the
    distance from the crossing to it."""
    radius, half, cells, n_expected = COARSE[name]
    v, surf = _patch(radius, half, cells, 1.0)
    n = 1_000_000
    rng = np.random.default_rng(int(radius + half + cells))
    k = rng.integers(0, len(v), n)
    e = rng.integers(0, 3, n)
    b = np.zeros((n, 3))
    b[np.arange(n), e] = rng.uniform(0.35, 0.65, n)
    b[np.arange(n), (e + 1) % 3] = 1.0 - b[np.arange(n), e]
    b[np.arange(n), (e + 2) % 3] = rng.uniform(0.001, 0.1, n)
    b /= b.sum(1, keepdims=True)
    t = v[k].astype(np.float64)
    p = np.einsum("ij,ijk->ik", b, t)
    # the proxy's sphere: the centre, and a radius in the middle of the facets'
    q = v.reshape(-1, 3).astype(np.float64)
    x = np.linalg.lstsq(np.c_[2 * q, np.ones(len(q))], (q * q).sum(1), rcond=None)[0][:3]
    g = np.cross(t[:, 1] - t[:, 0], t[:, 2] - t[:, 0])
    inner = np.abs(((t[:, 0] - x) * g).sum(1) / np.linalg.norm(g, axis=1)).min()
    r = 0.5 * (inner + np.linalg.norm(q - x, axis=1).max())
    nrm = p - x
    rho = np.linalg.norm(nrm, axis=1)
    nrm /= rho[:, None]
    s2 = (1.0 - rng.uniform(0.24, 0.3, n) ** 2) * (r / rho) ** 2
    c = np.sqrt(np.maximum(0.0, 1.0 - s2)) * rng.choice([-1.0, 1.0], n)
    side = rng.standard_normal((n, 3))
    side -= (side * nrm).sum(1, keepdims=True) * nrm
    side /= np.linalg.norm(side, axis=1, keepdims=True)
    d = (c[:, None] * nrm + np.sqrt(1 - c * c)[:, None] * side).astype(np.float32)
    o = (p - d * rng.uniform(0.2, 1.0, (n, 1)) * radius).astype(np.float32)
    k = np.zeros(n, np.int32)
    t_hit = np.zeros(n)
    lib.nearest_tri(C.c_int64(len(v)), v.ctypes.data_as(C.c_void_p), None, C.c_int64(n),
                    *(a.ctypes.data_as(C.c_void_p) for a in (o, d)), None,
                    *(a.ctypes.data_as(C.c_void_p) for a in (k, t_hit)))
    on = k >= 0
    assert on.mean() > 0.3
    n_proxies, out, reach = _find(lib, v, surf, float(np.abs(v).max()) + radius, o[on], d[on],
                                  k[on], t_hit[on])
    assert n_proxies == n_expected
    if n_proxies:
        assert np.all(out != 0), (int((out == 0).sum()), len(out))
        assert 0.1 < reach <= 1.0


def _tiles(radius, half, cells, gap):
    """A square patch of a sphere (or a plane, radius 0) cut into 2 x 2 surfaces, `gap`
    apart, and a plane of one surface across the light that they send back."""
    tris, surf = [], []
    for i, x in enumerate((-1, 1)):
        for j, y in enumerate((-1, 1)):
            xs, ys = sorted((x * gap / 2, x * half)), sorted((y * gap / 2, y * half))
            if radius:
                t, _ = W._mesh_rect_tile(np.zeros(3), radius, *np.eye(3)[[2, 0, 1]], *xs, *ys,
                                         cells, cells)
            else:
                t = W._mesh_rectangle(np.array([xs[0], ys[0], 300.0]), *np.eye(3)[:2],
                                      xs[1] - xs[0], ys[1] - ys[0], cells, cells)
            tris.append(t)
            surf.append(np.full(len(t), 2 * i + j))
    t = W._mesh_rectangle(np.array([-half, -1.5 * half, -100.0]), *np.eye(3)[:2], 2.5 * half,
                          3 * half, 4, 4)
    return (np.concatenate(tris + [t]).astype(np.float32),
            np.concatenate(surf + [np.full(len(t), 4)]).astype(np.int32))


def _stack():
    """Five parallel planes with half of their triangles missing, so that a ray looks up
    cells whose triangles it misses."""
    t = [W._mesh_rectangle(np.array([0.0, 0.0, 15.0 * k]), *np.eye(3)[:2], 300.0, 300.0, 20, 20)
         for k in range(5)]
    t = [x[np.random.default_rng(k).random(len(x)) < 0.5] for k, x in enumerate(t)]
    return (np.concatenate(t).astype(np.float32),
            np.repeat(np.arange(5, dtype=np.int32), [len(x) for x in t]))


def _meshes(scene):
    return scene.tri_vertices, scene.tri_surface


SINGLE, APART = 0x10, 0x20
# surfaces, and the codes of their triangles
LEAVE = {
    "tiles_apart": (lambda: _tiles(500.0, 200.0, 5, 30.0), {SINGLE, APART}),
    "tiles_apart_coarse": (lambda: _tiles(500.0, 150.0, 2, 60.0), {SINGLE, APART}),
    "tiles_touching": (lambda: _tiles(500.0, 200.0, 5, 0.0), {SINGLE, 0}),
    "flats_apart": (lambda: _tiles(0.0, 200.0, 5, 30.0), {SINGLE, APART}),
    "flats_touching": (lambda: _tiles(0.0, 200.0, 5, 0.0), {SINGLE, 0}),
    "stack": (_stack, {SINGLE}),
    "rich1": (lambda: _meshes(W.rich1_scene(tiles_per_edge=8, flat_cells=(8, 6))), {SINGLE, APART}),
    "rich2": (lambda: _meshes(W.rich2_scene(hex_subdiv=6)), {SINGLE, 0}),
}


@pytest.mark.parametrize("name", sorted(LEAVE))
def test_a_ray_that_leaves_a_facet_finds_the_next_surface(lib, name):
    """Rays that start on a facet, in every direction (half of them at other
    triangles): the surface just left is passed over with its proxy or with the
    entry crossing, and the nearest triangle of any other surface is still found."""
    make, codes_expected = LEAVE[name]
    v, surf = make()
    v, surf = np.ascontiguousarray(v, np.float32), np.ascontiguousarray(surf, np.int32)
    n = min(200_000, 100_000_000 // len(v))
    rng = np.random.default_rng(len(v))
    at = lambda k: np.einsum("ij,ijk->ik", rng.dirichlet((0.6, 0.6, 0.6), n), v[k].astype(float))
    k = rng.integers(0, len(v), n).astype(np.int32)
    o = at(k).astype(np.float32)
    d = rng.standard_normal((n, 3))
    aimed = rng.random(n) < 0.5
    d[aimed] = (at(rng.integers(0, len(v), n)) - o)[aimed]
    d = (d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32)
    target, t_hit = np.zeros(n, np.int32), np.zeros(n)
    out, codes, used = np.zeros(n, np.uint8), np.zeros(len(v), np.uint32), C.c_int64()
    p = {a: x.ctypes.data_as(C.c_void_p) for a, x in
         dict(v=v, s=surf, o=o, d=d, k=k, target=target, t=t_hit, out=out, codes=codes).items()}
    lib.nearest_tri(C.c_int64(len(v)), p["v"], p["s"], C.c_int64(n), p["o"], p["d"], p["k"],
                    p["target"], p["t"])
    n_proxies = lib.proxy_leave(C.c_int64(len(v)), p["v"], p["s"],
                                C.c_double(float(np.abs(v).max())), C.c_int64(n), p["o"], p["d"],
                                p["k"], p["target"], p["t"], p["out"], p["codes"], C.byref(used))
    assert n_proxies > 0
    found = set((codes & (SINGLE | APART)).tolist())
    assert found == codes_expected, found
    lost = (target != -2) & (out == 0)
    assert not lost.any(), (int(lost.sum()), n, np.flatnonzero(lost)[:5])
    assert used.value > n / 20 and (target >= 0).mean() > 0.1 and ((out & 2) == 0).mean() > 0.3


def test_meshes_off_any_sphere_or_plane_use_the_bvh(lib):
    """A bent surface, a closed sphere and more surfaces than proxies: none."""
    v, _ = _patch(0.0, 100.0, 6, 1.0, 10.0)
    bent = v.copy()
    bent[..., 2] += 10.0 * np.sin(bent[..., 0] / 20.0)
    ball = W._orient(np.concatenate([s * W._sphere_point(
        np.zeros(3), 100.0, *np.eye(3)[[2, 0, 1]],
        *np.random.default_rng(0).uniform(-70, 70, (2, 300))).reshape(-1, 3, 3)
        for s in (1.0, -1.0)]), np.zeros(3), 100.0)[0].astype(np.float32)
    rng = np.random.default_rng(1)
    many = np.concatenate([v @ np.linalg.qr(rng.standard_normal((3, 3)))[0].astype(np.float32)
                           for _ in range(9)])
    surfs = (None, None, np.repeat(np.arange(9, dtype=np.int32), len(v)))
    for m, s in zip((bent, ball, many), surfs):
        m = np.ascontiguousarray(m, np.float32)
        none = np.zeros((0, 3), np.float32)
        assert _find(lib, m, s, 1000.0, none, none, np.zeros(0, np.int32))[0] == 0
