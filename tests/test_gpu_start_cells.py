"""Start cells of 1-D batches: batch sizes around the anchors' strides, with one
origin, some (fine anchors, rays match another anchor's origin), up to and beyond
half the anchors, and all different (coarse anchors and greedy descents)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import oracle as O  # noqa: E402
from paper_2608_17682_gb300 import api  # noqa: E402
from paper_2608_17682_gb300 import workloads as W  # noqa: E402

DEV = "cuda"


@pytest.fixture(scope="module")
def cloud():
    sc = W.make_scene("uniform", 3000, 2, 71)
    return O.OracleScene.from_workload_scene(sc), api.Scene.from_workload(sc)


@pytest.mark.parametrize("n", [1, 63, 64, 65, 4096, 4097, 9001, 270_001])
@pytest.mark.parametrize("origins", [1, 4, 9, 30, 40, 0])
def test_start_cells_of_a_batch(cloud, n, origins):
    osc, scene = cloud
    rng = np.random.default_rng(n + 7 * origins)
    k = origins or n
    eyes = rng.uniform(-0.2, 1.2, (k, 3)).astype(np.float32)
    o = eyes[np.sort(rng.integers(0, k, n))] if origins else eyes
    d = rng.normal(size=(n, 3))
    d = (d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32)
    cells, _, _ = api.trace_cells(scene, torch.as_tensor(o, device=DEV), torch.as_tensor(d, device=DEV),
                                  api.make_params(), max_cells=64)
    assert scene.get_error()[0] == 0
    pick = np.unique(np.linspace(0, n - 1, min(n, 4000)).astype(int))
    oc, _, _, flags = O.trace(osc, o[pick], d[pick], max_cells=64, params=O.make_params())
    ok = (flags & O.BAND_FLAGS) == 0
    assert np.array_equal(cells.cpu().numpy()[pick][ok], oc[ok])


@pytest.mark.parametrize("cams", [2, 9, 20])
def test_start_cells_of_a_batch_laid_out_as_images(cloud, cams):
    """An image table over a batch: each image's first ray is another camera's."""
    osc, scene = cloud
    rng = np.random.default_rng(cams)
    eyes = rng.uniform(-0.2, 1.2, (cams, 3)).astype(np.float32)
    w, h = 40, 9
    which = np.roll(np.repeat(np.arange(cams), w * h), 1)
    d = rng.normal(size=(len(which), 3))
    d = (d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32)
    cells, _, _ = api.trace_cells(scene, torch.as_tensor(eyes[which], device=DEV), torch.as_tensor(d, device=DEV),
                                  api.make_params(image_sizes=[(w, h)] * cams), max_cells=64)
    assert scene.get_error()[0] == 0
    oc, _, _, flags = O.trace(osc, eyes[which], d, max_cells=64, params=O.make_params())
    ok = (flags & O.BAND_FLAGS) == 0
    assert np.array_equal(cells.cpu().numpy()[ok], oc[ok])


@pytest.mark.parametrize("far", [0.0, 3.0, 1e4, 1e19])
def test_descent_among_equal_distances(far):
    """Lattice sites, all 26 neighbours: origins at cell corners, edges and faces have two to eight nearest sites, of
    which the lowest id counts. `far`: origins that far outside, whose distances FP32 hardly or no longer tells apart;
    there the cell's own key must be the least among its neighbours'."""
    k, n = 7, 5000
    ijk = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3)
    rng = np.random.default_rng(91)
    ids = rng.permutation(k**3)  # site of each lattice place
    step = np.array([s for s in np.ndindex(3, 3, 3) if s != (1, 1, 1)]) - 1
    rows = [None] * k**3
    for place, at in enumerate(ijk):
        nb = at + step
        nb = nb[((nb >= 0) & (nb < k)).all(1)]
        rows[ids[place]] = ids[(nb * [k * k, k, 1]).sum(1)]
    sites = np.empty((k**3, 3), np.float32)
    sites[ids] = ijk
    off = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    sc = W.Scene(sites, np.ones(k**3, np.float32), W.textures(k**3, 2, rng), off, np.concatenate(rows).astype(np.int32))
    scene = api.Scene.from_workload(sc)
    o = (0.5 * rng.integers(0, 2 * k - 1, (n, 3))).astype(np.float32)
    d = rng.normal(size=(n, 3))
    d = (d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32)
    o = o + np.float32(far) * np.sign(d) * (rng.random((n, 3)) < 0.5).astype(np.float32)
    cells = api.trace_cells(scene, torch.as_tensor(o, device=DEV), torch.as_tensor(d, device=DEV), api.make_params(),
                            max_cells=1)[0][:, 0].cpu().numpy()
    with np.errstate(over="ignore"):
        if far <= 3.0:  # exact in FP32
            d2 = ((o[:, None] - sites) ** 2).sum(2)
            assert np.array_equal(cells, d2.argmin(1))  # the first, so the lowest id
            return
        delta = np.float32(o[:, None] - sites).astype(np.float64)

        def key(i, j):  # FP32 distance as the kernel forms it: products and sums rounded once each
            x, y, z = delta[i, j]
            t = np.float32(z * z).astype(np.float64)
            t = np.float32(y * y + t).astype(np.float64)
            return float(np.float32(x * x + t)), j

        for i in range(0, n, 10):
            assert key(i, cells[i]) <= min(key(i, j) for j in rows[cells[i]])
