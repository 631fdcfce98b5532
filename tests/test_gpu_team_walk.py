"""The forward walk by teams of lanes (launches of few rays) against the walk
with a lane per ray: one launch of more rays than teams take, and the same rays
in small launches, bit for bit. The scene has a hub cell with more neighbours
than a team tests in one round, and the last record of the array is walked."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2608_17682_gb300 import api  # noqa: E402
from paper_2608_17682_gb300 import workloads as W  # noqa: E402

DEV = "cuda"


def hub_scene(seed):
    """A site amid 300 on a sphere around it (degree 300), and a uniform crowd outside."""
    rng = np.random.default_rng(seed)
    v = rng.normal(size=(300, 3))
    shell = 0.5 * v / np.linalg.norm(v, axis=1, keepdims=True)
    crowd = rng.uniform(-2, 2, (2500, 3))
    crowd = crowd[np.linalg.norm(crowd, axis=1) > 0.8]
    sites = np.concatenate([[[0.0, 0.0, 0.0]], shell, crowd]).astype(np.float32)
    off, idx = W.delaunay_csr(sites)
    assert off[1] - off[0] > 64
    n = len(sites)
    return W.Scene(sites, np.exp(rng.normal(-1, 1, n)).astype(np.float32), W.textures(n, 4, rng), off, idx)


@pytest.mark.parametrize("appearance,with_dist,dtype", [(0, False, "f32"), (0, True, "f16"), (1, False, "bf16"),
                                                        (1, True, "f32")])
def test_small_launches_equal_a_large_one(appearance, with_dist, dtype):
    sc = hub_scene(81)
    rng = np.random.default_rng(82)
    tvd = rng.normal(size=sc.tex.shape).astype(np.float32) if appearance else None
    scene = api.Scene.from_workload(sc, tex_dtype=dtype, tex_vd=tvd)
    n = 60_000
    o = rng.uniform(-1.5, 1.5, (n, 3)).astype(np.float32)
    o[: n // 2] *= 0.2  # half of the rays start in or next to the hub
    d = rng.normal(size=(n, 3))
    to = torch.as_tensor(o, device=DEV)
    td = torch.as_tensor((d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32), device=DEV)
    P = api.make_params(appearance=appearance, t_far=3.0)

    def render(a, b):
        res = torch.empty(b - a, 3, device=DEV)
        dist = torch.empty(b - a, 3, device=DEV) if with_dist else None
        rec = torch.zeros(62, b - a, dtype=torch.int64, device=DEV)
        rgb, T, steps = api.render_fwd(scene, to[a:b], td[a:b], P, residual=res, dist=dist, record=rec)
        return [x for x in (rgb, T, steps, res, dist) if x is not None] + [rec.t().contiguous()]

    whole = render(0, n)
    cuts = [0, 1, 3, 4, 100, 4196, 30_000, n]
    parts = [render(a, b) for a, b in zip(cuts, cuts[1:])]
    for k, x in enumerate(whole):
        assert torch.equal(torch.cat([p[k] for p in parts]), x)
    assert scene.get_error()[0] == 0


def lattice_scene(k, seed):
    """Sites of a cubic lattice, moved by a few FP32 roundings, with all 26 neighbours: cells meet eight in a corner."""
    rng = np.random.default_rng(seed)
    at = np.arange(k)
    ijk = np.stack(np.meshgrid(at, at, at, indexing="ij"), -1).reshape(-1, 3)
    sites = (ijk / k + rng.uniform(-2e-7, 2e-7, ijk.shape)).astype(np.float32)
    rows = []
    for c in ijk:
        lo, hi = np.maximum(c - 1, 0), np.minimum(c + 2, k)
        n = np.stack(np.meshgrid(*(np.arange(a, b) for a, b in zip(lo, hi)), indexing="ij"), -1).reshape(-1, 3)
        n = n[(n != c).any(1)]
        rows.append(rng.permutation((n[:, 0] * k + n[:, 1]) * k + n[:, 2]))
    off = np.concatenate([[0], np.cumsum([len(r) for r in rows])])
    n = len(sites)
    return W.Scene(sites, np.exp(rng.normal(-1, 1, n)).astype(np.float32), W.textures(n, 2, rng), off.astype(np.int64),
                   np.concatenate(rows).astype(np.int32))


def test_teams_take_the_same_of_planes_equal_within_rounding():
    """Rays through corners: seven crossings within some roundings of one another, whose comparisons depend on their
    order. The walk's cells and steps must be the single lane's."""
    k, n = 8, 120_000
    sc = lattice_scene(k, 83)
    rng = np.random.default_rng(84)
    corner = (rng.integers(1, k - 2, (n, 3)) + 0.5) / k
    d = rng.normal(size=(n, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    o = corner - rng.uniform(0.02, 0.5, (n, 1)) * d
    scene = api.Scene.from_workload(sc)
    to, td = (torch.as_tensor(x.astype(np.float32), device=DEV) for x in (o, d))
    P = api.make_params(T_eps=0.0)

    def walk(a, b):
        rec = torch.zeros(40, b - a, dtype=torch.int64, device=DEV)
        out = api.render_fwd(scene, to[a:b], td[a:b], P, record=rec)
        return [*out, rec.t().contiguous()]

    whole = walk(0, n)
    parts = [walk(a, a + 20_000) for a in range(0, n, 20_000)]
    differ = [int((torch.cat([p[i] for p in parts]) != x).reshape(n, -1).any(1).sum()) for i, x in enumerate(whole)]
    assert differ == [0, 0, 0, 0]
    single = api.trace_cells(scene, to[:20_000], td[:20_000], P, max_cells=32)  # (a lane per ray at any size)
    assert torch.equal(single[2], parts[0][2])
