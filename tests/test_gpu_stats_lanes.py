"""The statistics kernel gives a pixel a warp or four lanes, by the call's
pixels and batch length (a warp up to 32 pixels per sample of a batch of 64 or more
and up to 6080 pixels; up to 6080 from batches of 32 on; up to 1024 below).  Both
add the samples up in the same tree, so a pixel's statistics, event and decision
are the same bits in a call of many pixels and in calls of few."""
import ctypes

import numpy as np
import pytest
import torch

import scenegen as sg
from paper_2408_07996_gb300 import _lib as L
from parity import renderer_for

pytestmark = pytest.mark.gpu


def _step(state, pix, samples, k_base, spp_min, batch, spp_max, variant=0):
    """one detector step on a copy of the state: state, events, counts, means, undecided pixels"""
    n_total = state.shape[1]
    s = state.clone()
    ev = torch.full((n_total,), 9, dtype=torch.int8, device="cuda")
    spp = torch.full((n_total,), -1, dtype=torch.int32, device="cuda")
    mean = torch.full((n_total,), -1.0, device="cuda")
    und = torch.full((pix.numel(),), -1, dtype=torch.int32, device="cuda")
    p = [ctypes.c_void_p(s[i].data_ptr()) for i in range(6)]
    a = L.DetectArgs(L=samples.data_ptr(), pixels=pix.data_ptr(), n_pix=pix.numel(), n_total=n_total,
                     spp_r=samples.shape[1], reserved0=0, k_base=k_base, cur_n=p[0], cur_mean=p[1], cur_m2=p[2],
                     ref_n=p[3], ref_mean=p[4], ref_m2=p[5], events=ev.data_ptr(), spp_out=spp.data_ptr(),
                     mean_out=mean.data_ptr(), undecided=und.data_ptr(), eps=1e-3, C=0.2, alpha=0.05,
                     spp_min=spp_min, spp_batch=batch, spp_max=spp_max, variant=variant, se_mode=0,
                     stream=ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    n = ctypes.c_int64(-1)
    L.check(L.load().mcev_detect_batch_static(ctypes.byref(a), ctypes.byref(n)), None, "mcev_detect_batch_static")
    return s, ev, spp, mean, und[:n.value].sort().values


def _inputs(n, spp_min, count, first, spp_max):
    g = torch.Generator(device="cuda").manual_seed(n + count)
    samples = torch.exp(0.6 * torch.randn((n, count), generator=g, device="cuda"))
    samples[torch.rand((n, count), generator=g, device="cuda") < 0.01] = 0.0
    samples[0, 0] = float("inf")
    state = torch.zeros((6, n), dtype=torch.int32, device="cuda")
    m = torch.randn((2, n), generator=g, device="cuda") * 0.2
    state[0] = 0 if first else spp_min
    state[1] = m[0].view(torch.int32)
    state[2] = torch.full((n,), 0.3 * spp_min, device="cuda").view(torch.int32)
    state[3] = spp_max
    state[4] = m[1].view(torch.int32)
    state[5] = torch.full((n,), 0.3 * spp_max, device="cuda").view(torch.int32)
    return state, samples, torch.randperm(n, generator=g, device="cuda").to(torch.int32)


# (batch length, batches): the first batch of a frame, or a later window
@pytest.mark.parametrize("first", [True, False])
@pytest.mark.parametrize("batch,count", [(2, 3), (16, 5), (31, 4), (32, 4), (33, 3), (63, 2), (64, 7), (100, 2), (255, 2), (257, 1)])
def test_a_pixel_does_not_depend_on_the_calls_size(first, batch, count):
    spp_min = batch if first else 16
    spp_max = spp_min + batch * count + 5
    n = (1024 if batch < 32 else max(6080, 32 * batch)) + 1     # four lanes; the parts below: a warp per pixel
    k = spp_min if first else batch * count
    state, samples, pix = _inputs(n, spp_min, k, first, spp_max)
    whole = _step(state, pix, samples, 0 if first else spp_min, spp_min, batch, spp_max)
    edges = [0, 1, 8, 17, n // 2, n]
    undecided = []
    for a, b in zip(edges, edges[1:]):
        part = _step(state, pix[a:b], samples[a:b].contiguous(), 0 if first else spp_min, spp_min, batch, spp_max)
        at = pix[a:b].long()
        for x, y in zip(whole[:4], part[:4]):
            assert torch.equal(x[..., at], y[..., at])
        undecided.append(part[4])
    assert torch.equal(torch.cat(undecided).sort().values, whole[4])
    if not first and batch > 2:            # (six samples decide nothing)
        assert 0 < whole[4].numel() < n


@pytest.mark.parametrize("shape", [(1, 1), (5, 3), (13, 37), (61, 40)])
def test_frames_of_few_pixels_with_long_batches(shape):
    """Re-queueing where pixels have a warp each, with chunks of ragged sizes, against rounds of the whole image."""
    W, H = shape
    w = sg.workload("cornell64")
    outs = []
    for wavefront, host in ((0, 0), (1 << 12, 0), (1 << 12, 1)):
        r = renderer_for(w, W, H, wavefront=wavefront, host_rounds=host, spp_min=100)
        r.render_reference(0.0, 300)
        o = r.render_events(0.0, 1.0, 0.2, 0.05, 77, 900)
        assert o["stats"]["samples_used"] == int(o["spp"].sum()) and int(o["spp"].max()) <= 900
        outs.append([o[k].clone() for k in ("events", "spp", "mean")] + list(r.reference_arrays()))
        r.close()
    for o in outs[1:]:
        assert all(torch.equal(a, b) for a, b in zip(outs[0], o))


def test_one_pixels_samples_are_shared_by_a_warp():
    """8192 samples of one pixel: 286 us with four lanes, 40 us with a warp (GB300)."""
    state, samples, pix = _inputs(1, 8192, 8192, True, 8192)
    ms = []
    for _ in range(20):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        torch.cuda.synchronize()
        a.record()
        _step(state, pix, samples, 0, 8192, 8192, 8192)
        b.record()
        b.synchronize()
        ms.append(a.elapsed_time(b))
    # the call's own host work is part of it: the difference to a call of 32 samples
    state, samples, pix = _inputs(1, 32, 32, True, 32)
    base = []
    for _ in range(20):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        torch.cuda.synchronize()
        a.record()
        _step(state, pix, samples, 0, 32, 32, 32)
        b.record()
        b.synchronize()
        base.append(a.elapsed_time(b))
    print(np.median(ms), np.median(base))
    assert np.median(ms) - np.median(base) < 0.13
