"""Launch layout of the training samples (CPU): the images account for every
sample in order, keep rows of neighbouring samples, and are left out where the
samples are too sparse or the cameras too many."""
import numpy as np
import pytest

train = pytest.importorskip("paper_2608_17682_gb300.train")
from oracle import training as TR  # noqa: E402
from paper_2608_17682_gb300 import workloads as W  # noqa: E402


def cams(n, w, h, kind=0, **kw):
    return [W.look_at_camera(kind, w, h, W.orbit_eye(np.zeros(3), 3.0, 360.0 * k / n, 20.0), np.zeros(3), **kw)
            for k in range(n)]


@pytest.mark.parametrize("sizes,frac", [([(640, 416)] * 8, 0.49), ([(160, 120)] * 8, 0.43), ([(64, 48)], 1.0),
                                        ([(97, 61), (333, 40), (50, 200)], 0.8)])
def test_rows_of_samples_follow_image_rows(sizes, frac):
    cs = [c for s in sizes for c in cams(1, *s)]
    pool = sum(c.n_rays for c in cs)
    B = int(pool * frac)
    tiles = train.sample_tiles(cs, B)
    assert sum(w * h for w, h in tiles) == B and len(tiles) <= 64
    idx = TR.stratified_indices(pool, B, 5)
    first = np.concatenate([[0], np.cumsum([c.n_rays for c in cs])])
    at = 0
    for w, h in tiles:
        k = at + np.arange(w * h).reshape(h, w)
        at += w * h
        if h < 2:
            continue
        cam = np.searchsorted(first, idx[k], side="right") - 1
        assert (cam == cam[h // 2, w // 2]).mean() > 0.999  # a camera's own samples, but for one at either end
        c = cs[cam[h // 2, w // 2]]
        pix = idx[k] - first[cam[h // 2, w // 2]]
        # samples above one another come from next rows, within a pixel or two of the same column
        dx = np.diff(pix % c.w, axis=0)
        dx = (dx + c.w // 2) % c.w - c.w // 2
        assert np.median(np.abs(dx)) <= 1.5 / frac


def test_no_layout_for_sparse_samples_or_many_cameras():
    assert train.sample_tiles(cams(4, 100, 100), 4000) is None  # 10 samples a row
    # 4,029 samples of each camera: 63 rows of 63 and 60 more, two images each
    for n in (31, 32):
        tiles = train.sample_tiles(cams(n, 63, 64), n * 4029)
        assert tiles == [(63, 63), (60, 1)] * n
    assert train.sample_tiles(cams(33, 63, 64), 33 * 4029) is None
    assert train.sample_tiles(cams(70, 64, 64), 70 * 64 * 64) is None
