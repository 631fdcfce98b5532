"""The autograd entry point without a GPU, its kernel calls replaced: what it refuses and what it records."""
import pytest

torch = pytest.importorskip("torch")
fwad = pytest.importorskip("torch.autograd.forward_ad")

from paper_2608_17682_gb300 import api  # noqa: E402


class StandIn:
    n, R, has_tex_vd = 4, 2, False


@pytest.fixture
def calls(monkeypatch):
    """Records of the forward calls; colours are zero."""
    made = []

    def render_fwd(scene, o, d, params, out=None, record=None, **kw):
        made.append(record)
        out[0].zero_()

    monkeypatch.setattr(api, "render_fwd", render_fwd)
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
            api.render(*x, o, d, StandIn(), None)


@pytest.mark.parametrize("grad_mode", [True, False])
@pytest.mark.parametrize("needs", [True, False])
def test_a_walk_is_recorded_only_for_a_backward(calls, grad_mode, needs):
    sites, sigma, tex, o, d = arrays()
    sigma.requires_grad_(needs)
    with torch.set_grad_enabled(grad_mode):
        rgb = api.render(sites, sigma, tex, o, d, StandIn(), None)
    assert rgb.requires_grad == (grad_mode and needs)
    assert (calls[0] is not None) == (grad_mode and needs)
