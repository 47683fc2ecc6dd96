"""GPU parity of rays from everywhere on every kind of surface, against the
oracle (marked gpu): the surface proxies of meshes, the bounding spheres of
analytic tiles and the rectangle test answer for rays that meet surfaces from
either side, graze them, start on the far side of a sphere or far outside the
scene. Bars as in test_gpu_external.py, on the refined path: the fates and
surfaces are those of the FP32 trace in both, and FP32 positions of rays that
come 60 m are bounded by their coordinates' spacing (4e-3 mm at 60 m, times
1 / cos of a grazing incidence), which says nothing of the surfaces."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import oracle  # noqa: E402
from paper_2309_12496_gb300 import rich  # noqa: E402
from paper_2309_12496_gb300 import workloads as W  # noqa: E402

import parity as P  # noqa: E402
from test_gpu_external import _gpu_ext, _oracle_ext  # noqa: E402

SCENES = {
    "rich1": lambda: W.rich1_scene(meshed=True),
    "rich1_analytic": lambda: W.rich1_scene(meshed=False),
    "rich2": lambda: W.rich2_scene(meshed=True, hex_subdiv=6),
    "rich2_analytic": lambda: W.rich2_scene(meshed=False),
    "point": lambda: W.point_source_scene(),
    "point_meshed": lambda: W.point_source_scene(meshed=True),
    "two_mirror": lambda: W.two_mirror_scene(),
    "scint": lambda: W.scint_box_scene(),
}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2309_12496_gb300 import build
    build.build()
    oracle.build()


@pytest.mark.parametrize("name", sorted(SCENES))
@pytest.mark.parametrize("reach", [0.5, 8.0])
def test_rays_from_everywhere_match_the_oracle(name, reach):
    """Origins in a box of `reach` times the scene around it (inside and far
    outside), directions at points of the scene's box, so about half of the
    rays meet a surface; some along an axis."""
    scene = SCENES[name]()
    at = [scene.rects["origin"].astype(float)]
    if scene.n_triangles:
        at.append(scene.tri_vertices.reshape(-1, 3))
    for s in scene.spheres:
        at.append((s["center"] + s["radius"] * s["axis"])[None].astype(float))
    at = np.concatenate(at)
    lo, hi = at.min(0) - 50.0, at.max(0) + 50.0
    rng = np.random.default_rng(len(name))
    n = 40_000
    mid, half = 0.5 * (lo + hi), 0.5 * (hi - lo)
    o = (mid + half * 2 * reach * rng.uniform(-1, 1, (n, 3))).astype(np.float32)
    aim = mid + half * rng.uniform(-1, 1, (n, 3))
    d = aim - o
    axis = rng.random(n) < 0.05
    d[axis] = np.eye(3)[rng.integers(0, 3, int(axis.sum()))] * rng.choice([-1.0, 1.0], (int(axis.sum()), 1))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    arrays = {"x": o[:, 0], "y": o[:, 1], "z": o[:, 2], "lambda": rng.uniform(200, 600, n),
              "event": rng.integers(0, 3, n).astype(np.uint32),
              "track": rng.integers(0, 2**32, n, dtype=np.uint64).astype(np.uint32),
              "photon": np.arange(n, dtype=np.uint32)}
    arrays.update({"d" + k: d[:, i] for i, k in enumerate("xyz")})
    arrays = {k: v if v.dtype == np.uint32 else np.ascontiguousarray(v, np.float32)
              for k, v in arrays.items()}
    P.set_grid(scene.planes)
    ref = _oracle_ext(scene, arrays, 11, 3)
    ctx = rich.Context(0)
    ctx.init_geometry(scene)
    gpu = _gpu_ext(ctx, scene, arrays, 11, rich.PREC_REFINE64, 3)
    ctx.close()
    stats = P.compare(gpu, ref, None, P.TOL_UV_REFINE, name=f"everywhere_{name}_{reach}",
                      keys=(arrays["event"], arrays["track"], arrays["photon"]))
    assert stats["hits"] > 0


# the most staged nodes of RICH1 that fit in 227 KB beside 1024, 512 and 896 threads'
# state and the small tables, without the surface proxies' 512 bytes
@pytest.mark.parametrize("knobs,most", [
    ({}, 1575), (dict(block_threads=512), 1575), (dict(block_threads=1024), 1367),
    (dict(block_threads=896, wide_regs=1), 1419), (dict(block_threads=256), 1783)])
@pytest.mark.parametrize("precision", [rich.PREC_REFINE64, rich.PREC_FP32])
def test_staged_nodes_up_to_the_shared_memory(knobs, most, precision):
    """A number of staged nodes is taken up to what the shared memory holds and
    refused above it, and does not change what is traced."""
    scene = W.rich1_scene(meshed=True)
    ctx = rich.Context(0)
    ctx.init_geometry(scene)
    dt = rich.DeviceTracks(W.pion_tracks(30, seed=3))
    n = ctx.emit(dt, 0.0014, seed=4)
    out = rich.TraceOutputs(n, scene.pixels_per_event, len(scene.planes), 1, n)
    got = []
    for nodes in (-1, 1300, most - 4, most):
        ctx.emit(dt, 0.0014, seed=4)
        out.clear()
        ctx.trace(out, precision=precision, bvh_smem_nodes=nodes, **knobs)
        n_hits, _ = ctx.hits()
        got.append((np.sort(out.hits_numpy(n_hits), order=["event", "track", "photon"]),
                    out.fate.cpu().numpy().copy()))
    with pytest.raises(rich.RichError):
        ctx.trace(out, precision=precision, bvh_smem_nodes=most + 1, **knobs)
    ctx.close()
    assert len(got[0][0]) > 1000
    for hits, fate in got[1:]:
        np.testing.assert_array_equal(hits, got[0][0])
        np.testing.assert_array_equal(fate, got[0][1])


def test_staged_nodes_of_a_gradient():
    """The same limits hold for the gradient's forward pass."""
    scene = W.rich1_scene(meshed=True)
    ctx = rich.Context(0)
    ctx.init_geometry(scene)
    tracks = W.pion_tracks(30, seed=3)
    dt = rich.DeviceTracks(tracks)
    n = ctx.emit(dt, 0.0014, seed=4)
    planes = len(scene.planes)
    out = rich.TraceOutputs(n, scene.pixels_per_event, planes, 1, n)
    ctx.trace(out)
    n_hits, _ = ctx.hits()
    h = out.hits_numpy(n_hits)
    tg = torch.from_numpy(W.ring_targets(30, planes, h["track"].astype(np.int64), h["plane"],
                                         h["u"] + 1.0, h["v"])).cuda()
    th = W.nominal_theta(scene, 0.0014)
    th[8] = 2000.0                       # (no tiles to apply it to)
    res = {}
    for nodes in (-1, 1571, 1575):
        res[nodes] = ctx.trace_grad(dt, th, tg, out, seed=4, bvh_smem_nodes=nodes)
    with pytest.raises(rich.RichError):
        ctx.trace_grad(dt, th, tg, out, seed=4, bvh_smem_nodes=1576)
    ctx.close()
    loss, grad, used = res[-1]
    assert used > 500
    for nodes in (1571, 1575):
        # sums of up to 1e5 FP64 terms in another order
        assert res[nodes][0] == pytest.approx(loss, rel=1e-10) and res[nodes][2] == used
        np.testing.assert_allclose(res[nodes][1], grad, rtol=1e-8, atol=1e-8 * np.abs(grad).max())
