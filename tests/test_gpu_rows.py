"""Row kernels at the sizes where their access width or loop changes: texture
rows of even and odd resolution, in one chunk per lane, three and many, aligned
and not; losses over channel counts that are and are not multiples of four."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from oracle import training as TR  # noqa: E402
from paper_2608_17682_gb300 import _vt, api  # noqa: E402
from paper_2608_17682_gb300 import workloads as W  # noqa: E402

DEV = "cuda"


def at(x, shift):
    """x on the device, `shift` floats past an aligned address."""
    buf = torch.empty(x.size + shift, device=DEV)
    t = buf[shift:].view(x.shape)
    t.copy_(torch.as_tensor(x))
    return t


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("reg", [0, 1])
@pytest.mark.parametrize("R", [2, 3, 4, 6, 7, 8, 10, 16])
def test_texture_adam_and_regularisers(R, reg, shift):
    rng = np.random.default_rng(100 * R + reg)
    n = 517
    perm = rng.permutation(n).astype(np.int32)
    shape = (n, R, R, 3)
    p, m, v = rng.normal(size=shape), rng.normal(size=shape), rng.uniform(0.5, 2.0, size=shape)
    p, m, v = (x.astype(np.float32) for x in (p, m, v))
    g = rng.normal(size=(n, R, R, 4)).astype(np.float32)
    tp, tm, tv = at(p, shift), at(m, shift), at(v, shift)
    tperm, tg = torch.as_tensor(perm, device=DEV), torch.as_tensor(g, device=DEV)
    loss = torch.zeros(1, device=DEV)
    lam = 0.3
    _vt.vt_adam_step_tex_scene_order(n, R, tperm.data_ptr(), tg.data_ptr(), tp.data_ptr(), tm.data_ptr(), tv.data_ptr(),
                                     reg, lam, 1e-2, 0.9, 0.999, 1e-15, 7, loss.data_ptr(), api._stream())
    gu = np.empty(shape)
    gu[perm] = g[..., :3]
    zero = np.zeros(shape)
    if reg == 0:
        L, gr, _ = TR.texture_regularizers(p, zero, 0.0, lam)
    else:
        L, _, gr = TR.texture_regularizers(zero, p, lam, 0.0)
    rp, rm, rv = TR.adam(p, gu + gr, m, v, 1e-2, 0.9, 0.999, 1e-15, 7)
    # FP32 sums of under 2e6 terms of one sign in blocks: 1e-5; moments: a few roundings
    assert abs(loss.item() - L) <= 1e-5 * L
    for a, b in ((tp, rp), (tm, rm), (tv, rv)):
        assert np.abs(a.cpu().numpy() - b).max() <= 2e-6 * np.abs(b).max()
    # the separate regulariser kernel adds the same gradient
    acc, tq = at(np.zeros(shape, np.float32), shift), at(p, shift)
    args = (tq.data_ptr(), 0, 0.0, lam, acc.data_ptr(), 0) if reg == 0 else (0, tq.data_ptr(), lam, 0.0, 0, acc.data_ptr())
    _vt.vt_texture_regularizers(n, R, *args, loss.data_ptr(), api._stream())
    assert abs(loss.item() - L) <= 1e-5 * L
    assert np.abs(acc.cpu().numpy() - gr).max() <= 2e-6 * np.abs(gr).max()


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 1023, 1024])
def test_losses_at_ragged_sizes(n, shift):
    rng = np.random.default_rng(n)
    a, b = (rng.uniform(0, 1, (n, 3)).astype(np.float32) for _ in range(2))
    ta, tb, g = at(a, shift), at(b, shift), at(np.zeros((n, 3), np.float32), shift)
    loss = torch.empty(1, device=DEV)
    r = a.astype(np.float64) - b
    _vt.vt_l2_loss(n, ta.data_ptr(), tb.data_ptr(), g.data_ptr(), loss.data_ptr(), api._stream())
    assert abs(loss.item() - (r * r).mean()) <= 1e-6 * (r * r).mean()
    assert np.allclose(g.cpu().numpy(), 2 * r / (3 * n), rtol=1e-6, atol=1e-7 / n)
    _vt.vt_smooth_l1_loss(n, ta.data_ptr(), tb.data_ptr(), 0.05, g.data_ptr(), loss.data_ptr(), api._stream())
    L, gr = TR.smooth_l1(a, b, 0.05)
    assert abs(loss.item() - L) <= 1e-6 * L
    assert np.allclose(g.cpu().numpy(), gr, rtol=2e-6, atol=2e-6 / n)


@pytest.mark.parametrize("R", [2, 3, 5, 6, 8, 9])
def test_gradient_rows_in_user_order(R):
    """render_bwd's user-order rows are the scene-order ones, permuted, and leave the scratch clean."""
    sc = W.make_scene("uniform", 1001, R, 90 + R)
    scene = api.Scene.from_workload(sc)
    rng = np.random.default_rng(R)
    n = 3000
    to = torch.as_tensor(rng.uniform(0, 1, (n, 3)).astype(np.float32), device=DEV)
    d = rng.normal(size=(n, 3))
    td = torch.as_tensor((d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32), device=DEV)
    P = api.make_params()
    rgb = api.render_fwd(scene, to, td, P)[0]
    g = torch.as_tensor(rng.normal(size=(n, 3)).astype(np.float32), device=DEV)
    out = at(np.full((sc.n, R, R, 3), np.nan, np.float32), 1)  # not aligned: single floats
    for grad in (g, torch.zeros_like(g), g):
        gs, gsig, gt = api.render_bwd(scene, to, td, P, rgb, grad)
        again = api.render_bwd(scene, to, td, P, rgb, grad, out=(None, None, out))[2]
        cell, tex, _ = api.render_bwd_scene_order(scene, to, td, P, rgb, grad)
        perm = scene.permutation().long()
        # sums of a few hundred FP32 terms in another order
        for a, b in ((gt[perm], tex[..., :3]), (again[perm], tex[..., :3]), (gs[perm], cell[:, :3]),
                     (gsig[perm], cell[:, 3])):
            assert (a - b).abs().max() <= 1e-4 * b.abs().max()


# The losses' sums hold what FP64 sums of the channels hold: bits that an FP32 sum of a chunk or row loses (small terms
# beside a large one), and squares beyond FP32's range. The results are FP32: one rounding each of the mean's factor and
# of the sum, 2^-24 each, the mean's where there are several blocks a few more.
BITS = 2.2 * 2.0**-24


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("far", [False, True])
def test_loss_sums_keep_what_fp64_holds(far, shift):
    n = 1024
    r = np.full((n, 3), 0.99 * 2.0**-12, np.float32)
    r.reshape(-1)[::4] = 1.0
    if far:  # 1e40 / 3072 is an FP32 number, 1e40 is not
        r[700, 1] = -1e20
    tr, zero = at(r, shift), at(np.zeros((n, 3), np.float32), shift)
    r, loss = r.astype(np.float64), torch.empty(1, device=DEV)
    _vt.vt_l2_loss(n, tr.data_ptr(), zero.data_ptr(), 0, loss.data_ptr(), api._stream())
    assert abs(loss.item() - (r * r).mean()) <= BITS * (r * r).mean()
    _vt.vt_smooth_l1_loss(n, tr.data_ptr(), zero.data_ptr(), 2.0, 0, loss.data_ptr(), api._stream())
    L = TR.smooth_l1(r, 0 * r, 2.0)[0]  # its terms are FP32: half an ulp each
    assert abs(loss.item() - L) <= (BITS + 2.0**-24) * L


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("scale,lam", [(1.0, 1.0), (1e25, 1e-22), (1e-25, 1e32)])
@pytest.mark.parametrize("R", [2, 7, 8, 64])
def test_regulariser_sums_keep_what_fp64_holds(R, scale, lam, shift):
    """One cell, so one block. A row's first channels are large, the mean of each colour is zero."""
    p = np.full((1, R * R, 3), 2.0**-13, np.float32)
    p[0, 1::2] *= -1
    if R % 2:
        p[0, -1] = 0.0
    p[0, 0], p[0, 1] = 1.0, -1.0
    p = (p * np.float32(scale)).reshape(1, R, R, 3)
    tp, z = at(p, shift), torch.zeros(1, dtype=torch.int32, device=DEV)
    loss = torch.zeros(1, device=DEV)
    want = {0: TR.texture_regularizers(p, 0 * p, 0.0, lam)[0], 1: TR.texture_regularizers(0 * p, p, lam, 0.0)[0]}
    for reg in (0, 1):
        loss.zero_()
        _vt.vt_adam_step_tex_scene_order(1, R, z.data_ptr(), 0, tp.data_ptr(), 0, 0, reg, lam, 0.0, 0.9, 0.999, 1e-15, 1,
                                         loss.data_ptr(), api._stream())
        # besides: the weight and 1/R^2 in FP32, and in reg 0 the deviations from an FP32 mean of 2^-24 or so
        assert abs(loss.item() - want[reg]) <= 2 * BITS * want[reg]
        args = (tp.data_ptr(), 0, 0.0, lam) if reg == 0 else (0, tp.data_ptr(), lam, 0.0)
        _vt.vt_texture_regularizers(1, R, *args, 0, 0, loss.data_ptr(), api._stream())
        assert abs(loss.item() - want[reg]) <= 2 * BITS * want[reg]
