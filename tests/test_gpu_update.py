"""A refused scene update changes nothing, although its kernels are launched
before its check is read; the next good one goes through."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2608_17682_gb300 import _vt, api  # noqa: E402
from paper_2608_17682_gb300 import workloads as W  # noqa: E402

DEV = "cuda"


@pytest.mark.parametrize("half", [False, True])
@pytest.mark.parametrize("where", ["sites", "sigma", "negative"])
def test_refused_update_changes_nothing(where, half):
    wl = W.make_workload("tiny", n_sites=1500)
    scene = api.Scene.from_workload(wl.scene, half_offsets=half)
    o, d = (torch.as_tensor(x, device=DEV) for x in W.workload_rays(wl))
    P = api.make_params(**wl.params, img_w=64, img_h=64, n_images=1)
    before = api.render_fwd(scene, o, d, P)
    new = {"sites": torch.rand(1500, 3, device=DEV), "sigma": torch.rand(1500, device=DEV),
           "tex": torch.rand(1500, 4, 4, 3, device=DEV)}
    bad = {k: v.clone() for k, v in new.items()}
    if where == "negative":
        bad["sigma"][7] = -1.0
    else:
        bad[where].view(-1)[-1] = float("nan")
    for _ in range(2):
        with pytest.raises(_vt.VTError) as e:
            scene.update(**bad)
        assert e.value.status == _vt.VT_ERR_INVALID_ARG
        for a, b in zip(api.render_fwd(scene, o, d, P), before):
            assert torch.equal(a, b)
    scene.update(**new)
    fresh = W.Scene(*(new[k].cpu().numpy() for k in ("sites", "sigma", "tex")), wl.scene.offsets, wl.scene.indices)
    other = api.Scene.from_workload(fresh, half_offsets=half, keep_order=True)
    assert not torch.equal(api.render_fwd(scene, o, d, P)[0], before[0])
    # the graph is the old sites': walks on it are the same in any cell order
    assert torch.equal(api.render_fwd(scene, o, d, P)[0], api.render_fwd(other, o, d, P)[0])


def test_a_refused_update_leaves_one_on_another_stream_alone():
    """An update returns while its kernels run; a refused one on another stream must not stop them half way."""
    wl = W.make_workload("tiny", n_sites=2000)
    n, R = 2000, 64  # long rows: the texture pass of the first update is still on its way when the second one is checked
    scene = api.Scene(wl.scene.sites, wl.scene.sigma, torch.rand(n, R, R, 3, device=DEV), wl.scene.offsets,
                      wl.scene.indices, tex_vd=torch.rand(n, R, R, 3, device=DEV))
    o, d = (torch.as_tensor(x, device=DEV) for x in W.workload_rays(wl))
    P = api.make_params(**wl.params, appearance=1)
    bad = torch.full((n,), float("nan"), device=DEV)
    streams = [torch.cuda.Stream() for _ in range(2)]
    for k in range(20):
        new = [torch.rand(n, 3, device=DEV), torch.rand(n, device=DEV), torch.rand(n, R, R, 3, device=DEV),
               torch.rand(n, R, R, 3, device=DEV)]
        torch.cuda.synchronize()
        with torch.cuda.stream(streams[0]):
            scene.update(*new)
        with torch.cuda.stream(streams[1]), pytest.raises(_vt.VTError):
            scene.update(sigma=bad)
        torch.cuda.synchronize()
        got = api.render_fwd(scene, o, d, P)[0]
        scene.update(*new)
        assert torch.equal(got, api.render_fwd(scene, o, d, P)[0]), k
