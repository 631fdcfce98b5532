"""The autograd entry point without a GPU, its kernel calls replaced: what it refuses and what it records."""
import weakref

import pytest

torch = pytest.importorskip("torch")
fwad = pytest.importorskip("torch.autograd.forward_ad")

from paper_2608_17682_gb300 import api  # noqa: E402


class StandIn:
    n, R, has_tex_vd, updates = 4, 2, False, 0


@pytest.fixture
def calls(monkeypatch):
    """Records (as weak references) that the forward and backward calls got; colours and gradients are zero."""
    made = []

    def note(record):
        made.append(None if record is None else weakref.ref(record))

    def render_fwd(scene, o, d, params, out=None, record=None, **kw):
        note(record)
        out[0].zero_()

    def render_bwd(scene, *a, record=None, **kw):
        note(record)
        return torch.zeros(4, 3), torch.zeros(4), torch.zeros(4, 2, 2, 3)

    monkeypatch.setattr(api, "render_fwd", render_fwd)
    monkeypatch.setattr(api, "render_bwd", render_bwd)
    return made


def arrays():
    return torch.rand(4, 3), torch.rand(4), torch.rand(4, 2, 2, 3), torch.rand(16, 3), torch.rand(16, 3)


@pytest.mark.parametrize("grad_mode", [True, False])
@pytest.mark.parametrize("which", [0, 1, 2])
def test_a_tangent_is_refused(calls, grad_mode, which):
    """There is no forward-mode derivative: a dual input raises, and never comes out as a colour without a tangent."""
    sites, sigma, tex, o, d = arrays()
    x = [sites, sigma, tex]
    with fwad.dual_level(), torch.set_grad_enabled(grad_mode):
        x[which] = fwad.make_dual(x[which], torch.ones_like(x[which]))
        with pytest.raises((NotImplementedError, RuntimeError)):
            api.render(*x, o, d, StandIn(), api.make_params())


@pytest.mark.parametrize("grad_mode", [True, False])
@pytest.mark.parametrize("needs", [True, False])
def test_a_walk_is_recorded_only_for_a_backward(calls, grad_mode, needs):
    sites, sigma, tex, o, d = arrays()
    sigma.requires_grad_(needs)
    with torch.set_grad_enabled(grad_mode):
        rgb = api.render(sites, sigma, tex, o, d, StandIn(), api.make_params())
    assert rgb.requires_grad == (grad_mode and needs)
    assert (calls[0] is not None) == (grad_mode and needs)


def render(scene=None, params=None):
    sites, sigma, tex, o, d = arrays()
    return api.render(sites, sigma.requires_grad_(True), tex, o, d, scene or StandIn(), params or api.make_params())


def test_the_record_lives_as_long_as_the_saved_tensors(calls):
    rgb = render()
    rgb.sum().backward(retain_graph=True)
    rgb.sum().backward()
    assert calls[0] is calls[1] is calls[2]
    assert calls[0]() is None  # rgb and its node are still here


def test_hooks_of_saved_tensors_do_not_see_the_record(calls):
    packed = []

    def pack(t):
        packed.append(t.nbytes)
        return t.clone()

    with torch.autograd.graph.saved_tensors_hooks(pack, lambda t: t):
        rgb = render()
    assert sorted(packed) == [16 * 3 * 4] * 4  # o, d, rgb, residual
    rgb.sum().backward()
    assert calls[1] is None  # the residual that came back is another tensor: the backward searches


STEP = 8 * 16  # bytes of a step of the stand-in's 16 rays


def test_renders_that_live_together_share_the_bound(calls, monkeypatch):
    monkeypatch.setattr(api, "RECORD_BYTES", STEP * 40)
    monkeypatch.setattr(api, "ALL_RECORDS_BYTES", STEP * (40 + 40 + 30) + 1)
    for _ in range(2):  # what the first round held is given back
        alive = [render() for _ in range(5)]
        assert [r and r().shape[0] for r in calls] == [40, 40, 30, None, None]
        sum(x.sum() for x in alive).backward()
        del calls[:], alive


def fails_with_records(calls, monkeypatch, error):
    """render_bwd raises while it gets a record, or always where there never was one."""
    given, plain = [], api.render_bwd

    def render_bwd(*a, record=None, **kw):
        given.append(record is not None)
        if record is not None or not calls[0]:
            raise error()
        return plain(*a, **kw)

    monkeypatch.setattr(api, "render_bwd", render_bwd)
    return given


def no_room():
    return api.VTError(api._vt.VT_ERR_OOM)


def fault():
    return api.VTError(api._vt.VT_ERR_CUDA)


OOM = [no_room, torch.cuda.OutOfMemoryError]


@pytest.mark.parametrize("error", OOM)
def test_a_backward_without_room_gives_up_the_records(calls, monkeypatch, error):
    given = fails_with_records(calls, monkeypatch, error)
    first, second = render(), render()
    second.sum().backward()
    first.sum().backward()
    assert given == [True, False, False]
    assert calls[0]() is None and calls[1]() is None


@pytest.mark.parametrize("error", OOM + [fault])
def test_other_failures_stay(calls, monkeypatch, error):
    if error is not fault:
        monkeypatch.setattr(api, "RECORD_BYTES", 0)  # no records to give up
    given = fails_with_records(calls, monkeypatch, error)
    with pytest.raises((api.VTError, torch.cuda.OutOfMemoryError)):
        render().sum().backward()
    assert len(given) == 1


def test_a_changed_scene_or_parameter_leaves_the_record_out(calls, monkeypatch):
    """The backward walks the scene as it stands, as without a record; timing events are not part of the walk."""
    scene, params = StandIn(), api.make_params()
    seen = []
    for change in (lambda: None, lambda: setattr(scene, "updates", scene.updates + 1),
                   lambda: setattr(params, "T_eps", 0.5), lambda: params.walk_events.__setitem__(0, 8)):
        rgb = render(scene, params)
        change()
        rgb.sum().backward()
        seen.append(calls[-1] is not None)
    assert seen == [True, False, False, True]
