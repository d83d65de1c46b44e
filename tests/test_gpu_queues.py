"""The ray queues and the traversal's groups at the edges of their tiles: a
sample's radiance and decision signature depend on its pixel and index alone, so
a call of n paths must give the bits that the same paths give in calls of
other sizes."""
import pytest
import torch

import scenegen as sg
from paper_2408_07996_gb300.api import Renderer

pytestmark = pytest.mark.gpu

# paths per call around a warp (32), a traversal block's groups (128), one and
# several queue tiles (512 entries per step, at most 4096) and a full round of tiles
COUNTS = [1, 31, 32, 33, 129, 511, 513, 4095, 4097, 20001]
# never-moving geometry only, with one moving instance, with a TLAS
SPINS = {"static": 0, "one": 1, "tlas": 5}


@pytest.mark.parametrize("width", [2, 8])
@pytest.mark.parametrize("moving", sorted(SPINS))
def test_samples_do_not_depend_on_the_call(moving, width):
    sc = sg.icosphere_field(11, n_spheres=6, level=2, n_frames=3, dt=5e-3, env_w=64, env_h=32, n_spin=SPINS[moving])
    W, H = 173, 121
    r = Renderer(W, H)
    r.upload(sc)
    r.set_params(t_min=1e-3, max_depth=4, seed=5, bvh_width=width)
    pix = (torch.arange(max(COUNTS), dtype=torch.int32) * 7919) % (W * H)
    t = float(sc.key_times[1])
    # sample k of a pixel in calls of 3 samples per pixel against one per call
    whole = [r.trace_samples(t, pix, k, 1) for k in range(3)]
    for n in COUNTS:
        L, sig = r.trace_samples(t, pix[:n], 0, 3)
        for k in range(3):
            assert torch.equal(L[:, k], whole[k][0][:n, 0]), (n, k)
            assert torch.equal(sig[:, k], whole[k][1][:n, 0]), (n, k)
    assert whole[0][0].max() > 0
    r.close()


@pytest.mark.parametrize("spp_max", [31, 96, 257])
def test_round_window_only_changes_what_is_traced(spp_max):
    """Any window of batches per round gives the frame of one batch per round."""
    w = sg.workload("cornell64")
    out = {}
    for window in (1, 0, 64):
        r = Renderer(w.width, w.height)
        r.upload(w.scene)
        r.configure(w)
        r.set_params(batch_window=window)
        o = r.render_events(0.0, 1.0, w.C, w.alpha, 8, spp_max)
        out[window] = (o["events"].clone(), o["spp"].clone(), o["mean"].clone(), o["stats"])
        r.close()
    for window in (0, 64):
        for a, b in zip(out[1][:3], out[window][:3]):
            assert torch.equal(a, b)
        assert out[window][3]["samples_used"] == out[1][3]["samples_used"]
        assert out[window][3]["paths"] >= out[1][3]["paths"]


@pytest.mark.parametrize("W,H", [(1, 1), (15, 17), (16, 16), (33, 5), (5, 33), (257, 64), (640, 131)])
def test_every_pixel_is_queued_once(W, H):
    """The tiled first queue and the ordered re-queueing on ragged images and
    across the statistics kernel's and the re-queue's tile sizes: every pixel
    gets its samples, and the frame is the one of a queue of single chunks."""
    w = sg.workload("cornell64")
    outs = []
    for wavefront, host in ((0, 0), (4096, 0), (4096, 1)):
        r = Renderer(W, H)
        r.upload(w.scene)
        r.configure(w)
        r.set_params(wavefront=wavefront, host_rounds=host)
        r.render_reference(0.0, 24)
        assert bool((r.reference_arrays()[0] == 24).all())
        o = r.render_events(0.0, 1.0, w.C, w.alpha, w.spp_batch, 80)
        assert int(o["spp"].min()) >= w.spp_min and int(o["spp"].max()) <= 80
        assert o["stats"]["samples_used"] == int(o["spp"].sum())
        outs.append([o[k].clone() for k in ("events", "spp", "mean")])
        r.close()
    for o in outs[1:]:
        assert all(torch.equal(a, b) for a, b in zip(outs[0], o))
