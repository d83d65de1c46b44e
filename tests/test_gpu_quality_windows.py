"""Event-video distances around the limits of the window searches (15 columns
and rings per event, 64 rings per warp) and of the bit masks' words, against
the FP64 oracle's exact nearest neighbours: every count and squared distance
is an integer and must be equal."""
import numpy as np
import pytest
import torch

from oracle import quality as Q
from test_gpu_quality import _compare

pytestmark = pytest.mark.gpu


def _at(shape, *events):
    v = np.zeros(shape, np.int8)
    for t, y, x, p in events:
        v[t, y, x] = p
    return v


# one event against one at a given offset along each axis
@pytest.mark.parametrize("d", [1, 15, 16, 17, 31, 32, 33, 63, 64, 65, 90])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_one_event_at_distance(axis, d):
    shape = [3, 3, 3]
    shape[axis] = d + 3
    lo, hi = [1, 1, 1], [1, 1, 1]
    hi[axis] += d
    a, b = _at(shape, (*lo, 1)), _at(shape, (*hi, 1))
    g, o = _compare(a, b, tau2=d * d)
    assert g["matched_a"] == 1 and int(g["d2_a"].max()) == d * d
    _compare(a, -b)


@pytest.mark.parametrize("W", [1, 15, 31, 32, 33, 63, 64, 65, 97])
@pytest.mark.parametrize("density", [0.002, 0.2])
def test_random_videos_of_word_sized_rows(W, density):
    rng = np.random.default_rng(W)
    shape = (9, 23, W)
    v = [np.where(rng.random(shape) < density, rng.choice([-1, 1], shape), 0).astype(np.int8) for _ in range(2)]
    for tau2 in (0, 3, 300):
        _compare(v[0], v[1], tau2)


def test_more_far_events_than_the_list_holds():
    """Thousands of events whose nearest counterpart is far away or beyond the
    wide search: one polarity is matched by the exact transform, the other, with
    near neighbours, by the windows."""
    rng = np.random.default_rng(5)
    shape = (4, 40, 300)
    a = np.zeros(shape, np.int8)
    a[:, :, :120] = rng.random((4, 40, 120)) < 0.4
    b = _at(shape, (0, 0, 299, 1), (3, 39, 290, 1))
    near = rng.random((4, 40, 60)) < 0.1
    a[:, :, 200:260] -= near.astype(np.int8)
    b[:, :, 201:261] -= near.astype(np.int8)
    _compare(a, b)
    _compare(b, a, tau2=9)


@pytest.mark.parametrize("shift", [0, 1, 2, 3, 5, 13])
def test_unaligned_videos(shift):
    from paper_2408_07996_gb300.api import event_quality
    rng = np.random.default_rng(shift)
    shape = (3, 7, 77)
    v = [np.where(rng.random(shape) < 0.1, rng.choice([-1, 1], shape), 0).astype(np.int8) for _ in range(2)]
    dev = []
    for x in v:
        buf = torch.full((x.size + 16,), 1, dtype=torch.int8, device="cuda")   # not read: outside the video
        buf[shift:shift + x.size] = torch.from_numpy(x.reshape(-1)).cuda()
        dev.append(buf[shift:shift + x.size].view(shape))
    g, o = event_quality(*dev, tau2=2), Q.quality(*v, 2)
    for k in ("n_a", "n_b", "matched_a", "matched_b", "sq_diff"):
        assert g[k] == o[k]
