"""Where the event-video searches change path: two rings and 15 columns around an
event (settled up to d^2 = 9), cells of 32 columns x 8 rows x 8 frames for the
listed events, at most voxels / 512 + 16384 of them and 512 steps each, and the
exact transform for the sets beyond.  Counts and squared distances are integers
and equal the FP64 oracle's (or the closed form's)."""
import numpy as np
import pytest
import torch

from oracle import quality as Q
from test_gpu_quality import _compare, _gpu

pytestmark = pytest.mark.gpu

SEARCHES = 4        # kernels of a call that the searches settle; a set's transform adds 3 or 4


def _at(shape, *events):
    v = np.zeros(shape, np.int8)
    for t, y, x, p in events:
        v[t, y, x] = p
    return v


@pytest.mark.parametrize("d", [2, 3, 4, 5, 7, 8, 9, 10, 17, 23, 24, 25])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_distances_from_every_place_in_a_cell(axis, d):
    for o in range(0, 9 if axis < 2 else 33, 1 if axis < 2 else 4):
        shape = [3, 3, 3]
        shape[axis] = o + d + 2
        lo, hi = [1, 1, 1], [1, 1, 1]
        lo[axis] = o
        hi[axis] = o + d
        a, b = _at(shape, (*lo, 1)), _at(shape, (*hi, 1))
        g, _ = _compare(a, b, tau2=d * d)
        assert g["matched_a"] == g["matched_b"] == 1 and int(g["d2_a"].max()) == d * d


@pytest.mark.parametrize("step", [(2, 2, 0), (2, 2, 1), (1, 2, 2), (0, 0, 3), (3, 0, 0), (0, 3, 0), (3, 1, 0), (1, 3, 0),
                                  (0, 1, 3), (0, 3, 1), (2, 2, 2), (3, 0, 1), (3, 3, 3), (8, 8, 31), (7, 9, 33),
                                  (1, 0, 15), (0, 1, 16), (2, 2, 15)])
def test_diagonal_distances(step):
    for sign in (1, -1):
        lo = np.array([9, 10, 40])
        hi = lo + np.array([sign, 1, sign]) * step
        shape = (20, 24, 80)
        a, b = _at(shape, (*lo, -1)), _at(shape, (*hi, -1))
        g, _ = _compare(a, b, tau2=9)
        want = int((np.array(step) ** 2).sum())
        assert int(g["d2_a"].max()) == int(g["d2_b"].max()) == want
        assert g["matched_a"] == (want <= 9)


@pytest.mark.parametrize("over", [0, 1])
def test_as_many_far_events_as_the_list_holds(over):
    shape = (2, 100, 600)
    cap = int(np.prod(shape)) // 512 + 16384
    a = np.zeros(shape, np.int8)
    far_side = np.zeros(2 * 100 * 200, np.int8)
    far_side[np.random.default_rng(1).choice(far_side.size, cap - 1 + over, replace=False)] = 1
    a[:, :, :200] = far_side.reshape(2, 100, 200)
    b = _at(shape, (1, 20, 599, 1))               # its nearest is far too: cap + over listed in all
    g, _ = _compare(a, b)
    assert (g["kernel_launches"] > SEARCHES) == bool(over)
    _compare(b, a)


def test_opposite_ends_of_a_long_video_go_to_the_transform():
    """A search ring by ring would visit 740 rings for every event."""
    shape = (6000, 16, 24)
    rng = np.random.default_rng(2)
    a, b = np.zeros(shape, np.int8), np.zeros(shape, np.int8)
    a[:40] = rng.random((40, 16, 24)) < 0.01
    b[-40:] = rng.random((40, 16, 24)) < 0.01
    # the other polarity has its counterparts near by: the searches settle it
    a[1000:1010] -= (rng.random((10, 16, 24)) < 0.05).astype(np.int8)
    b[1010:1022] -= (rng.random((12, 16, 24)) < 0.05).astype(np.int8)
    g, _ = _compare(a, b)
    assert g["kernel_launches"] == SEARCHES + 2 * 4
    assert int(g["d2_a"].max()) > 5900 ** 2


def test_a_far_event_among_near_ones_does_not_need_the_transform():
    """One event in thousands whose nearest is some 200 steps away is searched for all the
    same: 25 rings of an empty volume, with occupied cell rows all around at one distance."""
    shape = (60, 420, 64)
    rng = np.random.default_rng(4)
    T, H, W = shape
    t, y, x = np.mgrid[:T, :H, :W]
    a, b = np.zeros(shape, np.int8), np.zeros(shape, np.int8)
    shell = ((t - 30) ** 2 + (y - 210) ** 2 > 200 ** 2) & (rng.random(shape) < 0.02)
    a[shell] = 1
    b[shell] = 1
    move = shell & (rng.random(shape) < 0.2)
    a[move] = 0
    a[30, 210, 32] = 1
    g, _ = _compare(a, b)
    assert g["kernel_launches"] == SEARCHES
    assert int(g["d2_a"].max()) > 199 ** 2


def test_many_far_events_spend_the_budget():
    """Thousands of events some 300 steps away: together more than voxels / 8 + 65536 steps."""
    shape = (2600, 24, 16)
    rng = np.random.default_rng(5)
    a, b = np.zeros(shape, np.int8), np.zeros(shape, np.int8)
    a[:20] = rng.random((20, 24, 16)) < 0.2
    b[-20:] = rng.random((20, 24, 16)) < 0.2
    g, _ = _compare(a, b)
    assert g["kernel_launches"] > SEARCHES


@pytest.mark.parametrize("shape", [(1, 3000, 2500), (1, 64, 16384), (3000, 2, 40), (64, 2000, 1)])
def test_few_targets_on_a_large_grid(shape):
    """A thousand scattered events against a single one in a corner."""
    rng = np.random.default_rng(3)
    T, H, W = shape
    n = 1000
    a = np.zeros(shape, np.int8)
    a.reshape(-1)[rng.choice(a.size, n, replace=False)] = 1
    b = _at(shape, (0, 0, 0, 1))
    g = _gpu(a, b, tau2=10000)
    t, y, x = (i.astype(np.int64) for i in np.nonzero(a))
    want = t * t + y * y + x * x
    np.testing.assert_array_equal(g["d2_a"].cpu().numpy()[a != 0], want)
    assert int(g["d2_b"].max()) == want.min() and g["matched_a"] == int((want <= 10000).sum())
    assert g["sum_dist_a"] == pytest.approx(np.sqrt(want.astype(np.float64)).sum(), rel=1e-12)
    assert g["gpu_ms"] < 20.0


@pytest.mark.parametrize("shift_a,shift_b", [(0, 1), (1, 2), (3, 0), (5, 14), (13, 7)])
def test_videos_of_different_alignment(shift_a, shift_b):
    from paper_2408_07996_gb300.api import event_quality
    rng = np.random.default_rng(shift_a)
    shape = (3, 7, 77)
    v = [np.where(rng.random(shape) < 0.1, rng.choice([-1, 1], shape), 0).astype(np.int8) for _ in range(2)]
    dev = []
    for x, shift in zip(v, (shift_a, shift_b)):
        buf = torch.full((x.size + 16,), 1, dtype=torch.int8, device="cuda")   # not read: outside the video
        buf[shift:shift + x.size] = torch.from_numpy(x.reshape(-1)).cuda()
        dev.append(buf[shift:shift + x.size].view(shape))
    g, o = event_quality(*dev, tau2=2, want_d2=True), Q.quality(*v, 2)
    for k in ("n_a", "n_b", "matched_a", "matched_b", "sq_diff"):
        assert g[k] == o[k]
    for key, x in (("d2_a", v[0]), ("d2_b", v[1])):
        got = g[key].cpu().numpy()
        np.testing.assert_array_equal(np.where(got[x != 0] == -2, -1, got[x != 0]), o[key])
        assert (got[x == 0] == -1).all()
