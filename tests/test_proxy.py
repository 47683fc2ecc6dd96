"""Surface proxies of meshed mirrors (rich_proxy), on the CPU: the ray side
compiled for the host beside the builder.

The property the trace relies on: a ray that meets a triangle is either left
to the BVH or finds that triangle in the cell of one of its crossings. Rays
are aimed at points of every kind of triangle, edges and corners included,
with FP32 origins and directions; grazing and distant ones too."""
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
#include <cstring>
using namespace rich;
extern "C" int proxy_find(int64_t nt, const float *v, const int32_t *surf, double extent, int64_t nr,
                          const float *o, const float *d, const int32_t *target, float t_max,
                          uint8_t *out, double *listed) {
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
            float t, b2, h2;
            bool sure, entering = false;
            if (proxy_misses(P, O[0], O[1], O[2], D[0], D[1], D[2], t_max)) continue;
            if ((int)k < R.n_planes) {
                cell[0] = proxy_plane(P, O[0], O[1], O[2], D[0], D[1], D[2], 1e-3f, t_max, t, sure);
            } else {
                cell[0] = proxy_sphere(P, O[0], O[1], O[2], D[0], D[1], D[2], 1e-3f, t_max, t, sure,
                                       entering, b2, h2);
                if (entering)
                    cell[1] = proxy_sphere_side(P, O[0] - P.cx, O[1] - P.cy, O[2] - P.cz, D[0], D[1],
                                                D[2], b2, h2, -1.0f, 1e-3f, t_max, t, true);
            }
            if (!sure) out[i] |= 2;
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
    out = np.zeros(n, np.uint8)
    listed = C.c_double()
    s = None if surf is None else np.ascontiguousarray(surf, np.int32)
    n_proxies = lib.proxy_find(C.c_int64(len(v)), v.ctypes.data_as(C.c_void_p),
                               None if s is None else s.ctypes.data_as(C.c_void_p),
                               C.c_double(float(np.abs(v).max())), C.c_int64(n),
                               o.ctypes.data_as(C.c_void_p), d.ctypes.data_as(C.c_void_p),
                               k.ctypes.data_as(C.c_void_p), C.c_float(3e38),
                               out.ctypes.data_as(C.c_void_p), C.byref(listed))
    assert n_proxies == {"rich1": 4, "rich2": 5}.get(name, 1)
    assert np.all(out != 0), (int((out == 0).sum()), np.flatnonzero(out == 0)[:5])
    if cos_min > 0.25 and dist < 5000:
        assert (out & 1).mean() > 0.5            # most by their cells


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
        listed = C.c_double()
        assert lib.proxy_find(C.c_int64(len(m)), m.ctypes.data_as(C.c_void_p),
                              None if s is None else s.ctypes.data_as(C.c_void_p),
                              C.c_double(1000.0), C.c_int64(0), None, None, None, C.c_float(1.0),
                              None, C.byref(listed)) == 0
