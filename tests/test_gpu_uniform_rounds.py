"""Uniform sampling decides at the cap only, so its rounds hold as many batches as the
window and the wavefront allow, and give the frame of one batch per round."""
import pytest
import torch

import scenegen as sg
from parity import renderer_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("host", [0, 1])
@pytest.mark.parametrize("wavefront,rounds", [(0, 5), (1 << 22, 1 + 32)])
def test_rounds_of_a_uniform_frame(host, wavefront, rounds):
    """16 samples, then windows of 16 batches of 16 up to 1024 (2 batches of 90k pixels fill 2^22 paths)."""
    out = {}
    for window in (0, 1):
        r = renderer_for(sg.workload("cornell64"), 346, 260, variant=3, host_rounds=host, wavefront=wavefront,
                         batch_window=window)
        r.render_reference(0.0, 32)
        o = r.render_events(0.0, 1.0, 0.2, 0.05, 16, 1024)
        out[window] = [o[k].clone() for k in ("events", "spp", "mean")]
        assert bool((o["spp"] == 1024).all()) and o["stats"]["paths"] == 346 * 260 * 1024
        assert o["stats"]["rounds"] == (64 if window else rounds)
        r.close()
    assert all(torch.equal(a, b) for a, b in zip(out[0], out[1]))
