"""Gradients of a batch against the sum, in 64 bits, of those of its rays taken one at a time: a ray alone is summed
with nothing, so this pins the sums over lanes (whole warps in one cell and texel, warps of mixed cells and texels,
ragged ends) and the two arrays that even and odd warps add to."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2608_17682_gb300 import api  # noqa: E402
from paper_2608_17682_gb300 import workloads as W  # noqa: E402

DEV = "cuda"


# rays: from one point, `spread` the tangent of their largest angle to the axis (0: all the same ray)
@pytest.mark.parametrize("n,spread", [(1, 0.0), (31, 0.0), (32, 0.0), (128, 1e-4), (161, 0.05), (200, 2.0)])
@pytest.mark.parametrize("appearance,R", [(0, 2), (0, 8), (1, 4)])
def test_batch_gradient_is_the_sum_over_its_rays(n, spread, appearance, R):
    sc = W.make_scene("surface", 1500, R, 71)
    rng = np.random.default_rng(72)
    tvd = rng.normal(size=sc.tex.shape).astype(np.float32) if appearance else None
    scene = api.Scene.from_workload(sc, tex_vd=tvd)
    d = np.array([1.0, 0.02, -0.03]) + spread * rng.uniform(-1, 1, (n, 3))
    d = (d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32)
    to = torch.tensor([[-1.7, 0.01, 0.02]], device=DEV).repeat(n, 1)
    td, g = torch.as_tensor(d, device=DEV), torch.as_tensor(rng.normal(size=(n, 3)).astype(np.float32), device=DEV)
    P = api.make_params(appearance=appearance)

    def grads(rows):
        o, dd, gg = (t[rows].contiguous() for t in (to, td, g))
        res = torch.empty(len(o), 3, device=DEV)
        rgb = api.render_fwd(scene, o, dd, P, residual=res)[0]
        vd = torch.empty(sc.tex.shape, device=DEV) if appearance else None
        out = list(api.render_bwd(scene, o, dd, P, rgb, gg, residual=res, tex_vd_out=vd))
        if not appearance:
            cell, tex, _ = api.render_bwd_scene_order(scene, o, dd, P, rgb, gg, residual=res)
            out += [cell.clone(), tex.clone()]
        return [t.double() for t in out + ([vd] if appearance else [])]

    got = grads(slice(None))
    want = [torch.zeros_like(t) for t in got]
    size = [torch.zeros_like(t) for t in got]
    for i in range(n):
        for t, w, s in zip(grads(slice(i, i + 1)), want, size):
            w += t
            s += t.abs()
    assert float(size[1].max()) > 0
    # FP32 sums of n addends in any order: n roundings of at most 2^-24 of the addends' magnitudes. A ray's own
    # values to a few roundings more (a cell entered twice in its sum: its own atomics' order)
    for t, w, s in zip(got, want, size):
        assert bool(((t - w).abs() <= (n + 8) * 2.0**-24 * s).all())
    assert scene.get_error()[0] == 0


@pytest.mark.parametrize("skip,density", [(2.0, 1.0), (0.0, 0.0)])
@pytest.mark.parametrize("appearance", [0, 1])
@pytest.mark.parametrize("order", ["user", "scene"])
def test_cells_without_colour_take_nothing_of_an_infinite_gradient(skip, density, appearance, order):
    """No cell is coloured: too little weight for the skip threshold, or no density."""
    sc = W.make_scene("uniform", 1500, 4, 73)
    rng = np.random.default_rng(74)
    n = 200
    tvd = rng.normal(size=sc.tex.shape).astype(np.float32) if appearance else None
    sc.sigma[:] *= density
    scene = api.Scene.from_workload(sc, tex_vd=tvd)
    d = rng.normal(size=(n, 3))
    to = torch.as_tensor(rng.uniform(0, 1, (n, 3)).astype(np.float32), device=DEV)
    td = torch.as_tensor((d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32), device=DEV)
    g = torch.full((n, 3), float("inf"), device=DEV)
    P = api.make_params(appearance=appearance, skip_weight=skip)
    rgb = api.render_fwd(scene, to, td, P)[0]
    if order == "user":
        vd = torch.empty(sc.tex.shape, device=DEV) if appearance else None
        maps = [api.render_bwd(scene, to, td, P, rgb, g, tex_vd_out=vd)[2], vd]
    else:
        maps = api.render_bwd_scene_order(scene, to, td, P, rgb, g)[1:]
    for x in maps:
        assert x is None or not x.any()


def test_cell_sums_of_a_scene_of_more_than_32_bits_of_texels():
    """A row of 2^20 + 1 slabs with 64x64 textures (110 GB). 2^26 times the same ray: a running FP32 sum of the rays'
    density gradients, in an array each for odd and even warps, stops growing at 2^24 addends; one of whole warps' sums,
    2^20 each, is off by 2^20 roundings of 2^-25 at most."""
    free = torch.cuda.mem_get_info()[0]
    if free < 140 << 30:
        pytest.skip("needs 140 GB of device memory")
    n, R, rays = (1 << 20) + 1, 64, 1 << 26
    x = torch.arange(n, device=DEV)
    sites = torch.stack([x.float(), 0 * x.float(), 0 * x.float()], 1)
    off = torch.clamp(2 * torch.arange(n + 1, device=DEV) - 1, 0, 2 * (n - 1))
    idx = torch.stack([x - 1, x + 1], 1).reshape(-1)
    idx = idx[(idx >= 0) & (idx < n)].int()
    tex = torch.zeros(n, R, R, 3, device=DEV)
    scene = api.Scene(sites, torch.full((n,), 3.0, device=DEV), tex, off, idx, tex_dtype="f16")
    del tex, x
    torch.cuda.empty_cache()
    P = api.make_params(skip_weight=2.0)  # no colours: the background shines through
    to = torch.tensor([[777_000.1, 0.0, 0.0]], device=DEV).repeat(rays, 1)
    td = torch.tensor([[1.0, 0.0, 0.0]], device=DEV).repeat(rays, 1)
    rgb = api.render_fwd(scene, to, td, P, want_steps=False)[0]

    def density_gradient(k):
        return api.render_bwd(scene, to[:k], td[:k], P, rgb[:k], torch.ones(k, 3, device=DEV), need=(True, True, False))[1]

    one, all_ = density_gradient(1).double(), density_gradient(rays).double()
    assert int((one != 0).sum()) > 1
    assert bool(((all_ - rays * one).abs() <= rays * (one.abs() * 2.0**20 * 2.0**-25)).all())
    scene.close()
