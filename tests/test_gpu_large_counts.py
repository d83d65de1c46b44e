"""Sample counts above 2^24, where FP32 holds only every second integer.  A
pixel whose count cannot reach the cap is never written, so the call has to
fail instead of returning with what the output held before; counts that FP32
holds are rendered."""
import pytest
import torch

import scenegen as sg
from paper_2408_07996_gb300 import McevError
from parity import renderer_for

pytestmark = pytest.mark.gpu

HELD, NOT_HELD = (1 << 24) + 2, (1 << 24) + 1


@pytest.mark.parametrize("host", [0, 1])
def test_counts_that_fp32_does_not_hold_are_refused(host):
    r = renderer_for(sg.workload("cornell64"), 2, 1, host_rounds=host)
    with pytest.raises(McevError, match="undecided"):
        r.render_mean(0.0, NOT_HELD)
    with pytest.raises(McevError, match="undecided"):
        r.render_reference(0.0, NOT_HELD)
    # a frame that starts with a count that is held and ends at one that is not
    r.render_reference(0.0, 64)
    r.set_params(variant=3)
    with pytest.raises(McevError, match="undecided"):
        r.render_events(0.0, 1.0, 0.2, 0.05, 1 << 20, NOT_HELD)
    # the context stays usable
    assert bool(torch.isfinite(r.render_mean(0.0, 64)).all())
    r.close()


@pytest.mark.parametrize("host", [0, 1])
def test_counts_that_fp32_holds_are_rendered(host):
    r = renderer_for(sg.workload("cornell64"), 2, 1, host_rounds=host)
    few, many = r.render_mean(0.0, 1 << 18), r.render_mean(0.0, HELD)
    # ln(L + eps) lies between ln(1e-3) and about 3, so its deviation is below 5 and 0.1 ten standard errors at 2^18
    assert float((few - many).abs().max()) < 0.1
    r.render_reference(0.0, HELD)
    n, mean, _ = r.reference_arrays()
    assert bool((n == HELD).all()) and torch.equal(mean, many)
    r.close()
