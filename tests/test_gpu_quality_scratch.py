"""Scratch of mcev_event_quality near a memory limit.  The transform alone needs 8
bytes per voxel and its envelope stacks; the searches' event bits are not kept
beside it where there is no room, and narrow videos need no more than wide
ones."""
import ctypes as C

import numpy as np
import pytest
import torch

from oracle import quality as Q
from paper_2408_07996_gb300 import McevError
from paper_2408_07996_gb300 import _lib as L

pytestmark = pytest.mark.gpu


class Limited:
    """A context whose allocator hands out at most `limit` bytes at a time."""

    def __init__(self, limit):
        self.limit, self.live, self.peak = limit, {}, 0
        self.lib, self.ctx = L.load(), C.c_void_p()
        assert self.lib.mcev_create(C.byref(self.ctx), 0, 1, 1) == 0

        def alloc(n, _):
            if sum(self.live.values()) + n > self.limit:
                return None
            p = torch.cuda.caching_allocator_alloc(int(n), 0, torch.cuda.current_stream().cuda_stream)
            self.live[p] = n
            self.peak = max(self.peak, sum(self.live.values()))
            return p

        def free(p, _):
            del self.live[p]
            torch.cuda.caching_allocator_delete(p)

        self.cb = L.ALLOC_FN(alloc), L.FREE_FN(free)
        assert self.lib.mcev_set_allocator(self.ctx, *self.cb, None) == 0

    def quality(self, a, b, tau2=3):
        T, H, W = a.shape
        dev = [torch.from_numpy(v).cuda() for v in (a, b)]
        q = L.Quality()
        L.check(self.lib.mcev_event_quality(self.ctx, C.c_void_p(dev[0].data_ptr()), C.c_void_p(dev[1].data_ptr()),
                                            W, H, T, tau2, None, None, C.byref(q)), self.ctx, "mcev_event_quality")
        return q.as_dict()

    def close(self):
        torch.cuda.synchronize()
        self.lib.mcev_destroy(self.ctx)
        assert not self.live


def _transform_bytes(W, H, T):
    """two volumes and the envelope stacks of the longer column pass, and 64 KiB for the counters"""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    stack = 0
    for lines, length in ((T * W, H), (H * W, T)):
        if length > 1:
            stack = max(stack, min((lines + 255) // 256, sms * 8) * 256 * length * 8)
    up = lambda x: (x + 255) // 256 * 256  # noqa: E731
    return 2 * up(4 * W * H * T) + up(stack) + (64 << 10)


def _far_apart(shape):
    """more far events than the list holds"""
    T, H, W = shape
    a, b = np.zeros(shape, np.int8), np.zeros(shape, np.int8)
    a[:, :, :W // 4] = np.random.default_rng(1).random((T, H, W // 4)) < 0.3
    b[0, 0, W - 1] = b[T - 1, H - 1, W - 2] = 1
    return a, b


def _same(g, o):
    for k in ("n_a", "n_b", "matched_a", "matched_b", "sq_diff"):
        assert g[k] == o[k], k
    for k in ("sum_dist_a", "sum_dist_b", "pscd", "f1"):
        assert g[k] == pytest.approx(o[k], rel=1e-12)


def test_the_transform_fits_where_it_alone_fits():
    a, b = _far_apart((200, 100, 40))
    o = Q.quality(a, b, 3)
    c = Limited(_transform_bytes(40, 100, 200))
    for _ in range(2):                              # the second call finds the transform's scratch in the way
        g = c.quality(a, b)
        assert g["kernel_launches"] > 4
        _same(g, o)
    c.close()
    c = Limited(_transform_bytes(40, 100, 200) // 2)
    with pytest.raises(McevError, match="OOM"):
        c.quality(a, b)
    _same(c.quality(a[:9, :9], b[:9, :9]), Q.quality(a[:9, :9], b[:9, :9], 3))      # still usable
    c.close()


@pytest.mark.parametrize("shape", [(600, 500, 1), (1, 3000, 1), (3000, 1, 1), (500, 300, 2)])
def test_narrow_videos_need_no_more_than_the_transform_did(shape):
    rng = np.random.default_rng(2)
    a, b = (np.where(rng.random(shape) < 2e-3, rng.choice([-1, 1], shape), 0).astype(np.int8) for _ in range(2))
    T, H, W = shape
    c = Limited(1 << 40)
    _same(c.quality(a, b), Q.quality(a, b, 3))
    # (the list of far events: 128 KiB + 1/64 byte per voxel)
    assert c.peak <= _transform_bytes(W, H, T) + (256 << 10)
    c.close()


def test_device_time_does_not_cover_the_allocations():
    import time
    a, b = _far_apart((200, 100, 40))
    c = Limited(1 << 40)
    first = c.cb[0]

    def slow(n, user):
        time.sleep(0.1)
        return first(n, user)

    c.slow = L.ALLOC_FN(slow)
    assert c.lib.mcev_set_allocator(c.ctx, c.slow, c.cb[1], None) == 0
    g = c.quality(a, b)                             # one allocation is between the searches and the transform
    assert g["kernel_launches"] > 4 and 0.0 < g["gpu_ms"] < 50.0
    c.close()
