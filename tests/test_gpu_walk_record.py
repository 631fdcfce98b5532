"""Backward along the forward's walk record against the backward that searches:
records that hold every step, some (the other rays are searched) and none, for
both appearances, with and without the distortion loss, in image and 1-D layout,
with rays that miss the clip box."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2608_17682_gb300 import api  # noqa: E402
from paper_2608_17682_gb300 import workloads as W  # noqa: E402

DEV = "cuda"


def close(a, b):
    """Equal up to the order of the sums: FP32 sums of up to some thousand terms of either sign, so about 1e-6 of an
    entry's terms; 1e-4 of the entry, floored at 1e-4 of the largest entry, leaves room for cancellation."""
    a, b = a.double(), b.double()
    return bool(((a - b).abs() <= 1e-4 * torch.maximum(b.abs(), 1e-3 * b.abs().max()) + 1e-12).all())


@pytest.mark.parametrize("steps", [0, 1, 5, 47])
@pytest.mark.parametrize("appearance,with_dist,dtype", [(0, False, "f32"), (0, True, "f16"), (1, False, "bf16"),
                                                        (1, True, "f32")])
@pytest.mark.parametrize("layout", ["image", "1d"])
def test_recorded_backward_matches_the_searching_one(steps, appearance, with_dist, dtype, layout):
    sc = W.make_scene("surface", 3000, 4, 61)
    rng = np.random.default_rng(62)
    tvd = rng.normal(size=sc.tex.shape).astype(np.float32) if appearance else None
    scene = api.Scene.from_workload(sc, tex_dtype=dtype, tex_vd=tvd)
    w, h = 61, 45
    o, d = W.frustum_rays(W.orbit_eye(np.zeros(3), 3.0, 40.0, 20.0), np.zeros(3), w, h, rng)
    to, td = torch.as_tensor(o, device=DEV), torch.as_tensor(d, device=DEV)
    n = len(o)
    kw = dict(img_w=w, img_h=h, n_images=1) if layout == "image" else {}
    P = api.make_params(appearance=appearance, use_clip_box=True, clip_lo=(-0.8, -0.8, -0.8), clip_hi=(0.8, 0.8, 0.8),
                        **kw)
    g = torch.as_tensor(rng.normal(size=(n, 3)).astype(np.float32), device=DEV)
    gd = torch.as_tensor(rng.normal(size=n).astype(np.float32), device=DEV) if with_dist else None
    res = torch.empty(n, 3, device=DEV)
    dist = torch.empty(n, 3, device=DEV) if with_dist else None
    plain = api.render_fwd(scene, to, td, P, residual=res, dist=dist)
    # what the forward does not write holds cells that the scene does not have
    rec = torch.full((steps + 2, n), -2, dtype=torch.int64, device=DEV)
    rgb, T, count = api.render_fwd(scene, to, td, P, residual=res, dist=dist, record=rec)
    for a, b in zip(plain, (rgb, T, count)):
        assert torch.equal(a, b)
    assert int(count.min()) == 0 and int(count.max()) > 5
    kwb = dict(residual=res, dist=dist, grad_dist=gd)
    vd = [torch.empty(sc.tex.shape, device=DEV) if appearance else None for _ in range(2)]
    want = api.render_bwd(scene, to, td, P, rgb, g, tex_vd_out=vd[0], **kwb)
    got = api.render_bwd(scene, to, td, P, rgb, g, tex_vd_out=vd[1], record=rec, **kwb)
    assert all(close(a, b) for a, b in zip(got, want))
    assert not appearance or close(vd[1], vd[0])
    cell, tex, _ = api.render_bwd_scene_order(scene, to, td, P, rgb, g, record=rec, **kwb)
    perm = scene.permutation().long()
    assert close(cell[:, :3], want[0][perm]) and close(cell[:, 3], want[1][perm])
    assert close(tex[..., :3], want[2][perm])
    assert scene.get_error()[0] == 0


@pytest.mark.parametrize("layout", [{}, {"image_sizes": [(25, 12), (20, 10)]}])
@pytest.mark.parametrize("steps", [0, 3, 4, 5, 20])
def test_record_of_rays_stopped_by_max_steps(steps, layout):
    sc = W.make_scene("uniform", 2000, 2, 63)
    scene = api.Scene.from_workload(sc)
    rng = np.random.default_rng(64)
    n = 500
    to = torch.as_tensor(rng.uniform(0.3, 0.7, (n, 3)).astype(np.float32), device=DEV)
    d = rng.normal(size=(n, 3))
    td = torch.as_tensor((d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32), device=DEV)
    P = api.make_params(T_eps=0.0, max_steps=4, **layout)
    rec = torch.full((steps + 2, n), -2, dtype=torch.int64, device=DEV)
    rgb = api.render_fwd(scene, to, td, P, record=rec)[0]
    g = torch.as_tensor(rng.normal(size=(n, 3)).astype(np.float32), device=DEV)
    want = api.render_bwd(scene, to, td, P, rgb, g)
    got = api.render_bwd(scene, to, td, P, rgb, g, record=rec)
    assert scene.get_error()[0] == api._vt.VT_ERR_MAX_STEPS
    assert all(close(a, b) for a, b in zip(got, want))


def test_record_is_left_out_where_it_does_not_fit():
    n = api.RECORD_BYTES // (8 * 10) + 1  # one ray more than 8 steps and the two ends have room for
    assert api.walk_record(0, DEV) is None and api.walk_record(n, "meta") is None
    assert api.walk_record(n - 1, "meta").shape == (10, n - 1)
    assert api.walk_record(100, "meta").shape == (api.RECORD_STEPS + 2, 100)


@pytest.mark.parametrize("room", [0, 12, 70, 10_000])
def test_gradients_do_not_depend_on_the_room_for_records(monkeypatch, room):
    """Three renders alive before one backward, under bounds that hold some steps of the first record to all of all."""
    sc = W.make_scene("uniform", 2000, 3, 65)
    scene = api.Scene.from_workload(sc)
    rng = np.random.default_rng(66)
    n = 700
    P = api.make_params(t_far=2.0)
    leaves = [torch.as_tensor(x, device=DEV).requires_grad_(True) for x in (sc.sites, sc.sigma, sc.tex)]
    rays = []
    for _ in range(3):
        d = rng.normal(size=(n, 3))
        rays.append([torch.as_tensor(x.astype(np.float32), device=DEV)
                     for x in (rng.uniform(0, 1, (n, 3)), d / np.linalg.norm(d, axis=1, keepdims=True))])
    monkeypatch.setattr(api, "RECORD_BYTES", 0)
    want = [sum(g) for g in zip(*(torch.autograd.grad(api.render(*leaves, o, d, scene, P).square().sum(), leaves)
                                  for o, d in rays))]
    monkeypatch.undo()
    monkeypatch.setattr(api, "ALL_RECORDS_BYTES", 8 * n * room)
    got = torch.autograd.grad(sum(api.render(*leaves, o, d, scene, P).square().sum() for o, d in rays), leaves)
    assert all(close(a, b) for a, b in zip(got, want))


def test_an_update_between_forward_and_backward():
    """The backward walks the new sites, with or without room for a record."""
    sc = W.make_scene("uniform", 2000, 2, 67)
    rng = np.random.default_rng(68)
    n = 500
    d = rng.normal(size=(n, 3))
    o, d = (torch.as_tensor(x.astype(np.float32), device=DEV)
            for x in (rng.uniform(0, 1, (n, 3)), d / np.linalg.norm(d, axis=1, keepdims=True)))
    moved = torch.as_tensor(sc.sites + rng.normal(0, 1e-3, sc.sites.shape).astype(np.float32), device=DEV)
    P, grads = api.make_params(), []
    for record in (True, False):
        scene = api.Scene.from_workload(sc)
        sigma = torch.as_tensor(sc.sigma, device=DEV).requires_grad_(record)
        if record:
            rgb = api.render(torch.as_tensor(sc.sites, device=DEV), sigma, torch.as_tensor(sc.tex, device=DEV), o, d,
                             scene, P)
            scene.update(sites=moved)
            grads.append(torch.autograd.grad(rgb.square().sum(), sigma)[0])
        else:
            res = torch.empty(n, 3, device=DEV)
            rgb = api.render_fwd(scene, o, d, P, residual=res)[0]
            scene.update(sites=moved)
            grads.append(api.render_bwd(scene, o, d, P, rgb, 2 * rgb, residual=res)[1])
    assert close(*grads)
