"""Render parameters of a Trainer (CPU, the kernel calls replaced): every form of "no layout" is taken, the caller's
own layout stays, and later changes of the parameters reach the steps."""
import numpy as np
import pytest

train = pytest.importorskip("paper_2608_17682_gb300.train")
torch = pytest.importorskip("torch")
from paper_2608_17682_gb300 import workloads as W  # noqa: E402

CAMS = [W.look_at_camera(0, 64, 48, W.orbit_eye(np.zeros(3), 3.0, 90.0 * k, 20.0), np.zeros(3)) for k in range(2)]
POOL = 2 * 64 * 48


@pytest.fixture
def trainer(monkeypatch):
    class Scene:
        def __init__(self, *a, **kw):
            assert not any(train.api.Walk._held.values())  # the record comes after the memory that is needed

        def permutation(self):
            return None

        def close(self):
            pass

    z = torch.zeros(POOL, 3)
    monkeypatch.setattr(train.api, "Scene", Scene)
    monkeypatch.setattr(train.api, "sigma_from_rho", torch.exp)
    monkeypatch.setattr(train.api, "generate_rays", lambda cams: (z, z, z[:, 0]))

    def make(**rp):
        return train.Trainer(np.zeros((5, 3)), np.zeros(5), np.zeros((5, 2, 2, 3)), np.zeros((5, 2, 2, 3)), CAMS, z, rp,
                             train.TrainConfig(rays_per_iter=POOL), device="cpu", offsets=np.zeros(6), indices=[])

    return make


@pytest.mark.parametrize("rp", [{}, {"image_sizes": None}, {"img_w": 0, "img_h": 0, "n_images": 0}, {"n_images": 1}])
def test_parameters_without_a_layout(trainer, rp):
    p = trainer(t_far=7.0, **rp).step_params
    assert (p.t_far, p.appearance, p.n_images, bool(p.image_sizes)) == (7.0, 1, 2, True)


@pytest.mark.parametrize("rp", [{"img_w": 64, "img_h": 48, "n_images": 2}, {"image_sizes": [(64, 96)]}])
def test_the_callers_layout_stays(trainer, rp):
    t = trainer(**rp)
    p = t.step_params
    assert (p.img_w, p.image_sizes, p.n_images) == (t.rparams.img_w, t.rparams.image_sizes, rp.get("n_images", 1))


def test_the_record_counts_while_the_trainer_lives(trainer):
    t = trainer()
    assert t.walk.record.nbytes == sum(train.api.Walk._held.values()) > 0
    del t
    assert not any(train.api.Walk._held.values())


def test_later_changes_reach_the_steps(trainer):
    t = trainer()
    t.rparams.T_eps = 0.25
    assert t.step_params.T_eps == 0.25 and t.step_params.image_sizes and not t.rparams.image_sizes
