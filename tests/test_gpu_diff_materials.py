"""Emission gradients of scenes with many materials: the kernels add up the
first 32 materials' contributions per block and send the others' to global
memory at once, so emitters lie on both sides of index 32 here."""
import numpy as np
import pytest
import torch

import oracle as O
import scenegen as sg
from diffref import emission_fd, oracle_means
from parity import per_sample, renderer_for

pytestmark = pytest.mark.gpu

SPP = 64
LIGHTS = (5, 31, 32, 40)


def _room():
    """textured_room with 41 materials and its four emitters at LIGHTS"""
    sc = sg.textured_room(seed=21, grid=40, tex_size=32)
    where = np.array([0, 1, 2, 3, *LIGHTS])
    sc.tri_material = where[np.asarray(sc.tri_material)].astype(np.int32)
    for name in ("mat_type", "mat_albedo", "mat_rough", "mat_emit", "mat_textured"):
        old = np.asarray(getattr(sc, name))
        new = np.zeros(max(LIGHTS) + 1, old.dtype)
        new[where] = old
        setattr(sc, name, new)
    return sg.Workload("room41", sc, 64, 48, [0.0, 1.0], spp_min=16, spp_batch=16, spp_max=64, C=0.2, alpha=0.05,
                       max_depth=3, seed=4, t_min=6e-4), where


def _emission_grad(r, n_mat, g):
    ge = torch.zeros(n_mat, device="cuda")
    r.backward(0.0, SPP, g, None, ge)
    return ge.double().cpu().numpy()


def test_emission_gradients_on_both_sides_of_the_block_sums():
    w, where = _room()
    n = w.width * w.height
    pix = np.arange(n, dtype=np.int32)
    osc = O.OracleScene(w.scene)
    p = O.params_of(w)
    r = renderer_for(w)
    r.set_emission(torch.from_numpy(np.asarray(w.scene.mat_emit, np.float32)).cuda())
    keep = per_sample(r, osc, p, 0.0, pix, 0, SPP, w.eps)["match"].all(axis=1)
    assert keep.mean() > 0.9
    gw = (np.random.default_rng(6).normal(size=n) * keep).astype(np.float32)
    g = torch.from_numpy(gw).view(w.height, w.width).cuda()
    ge = _emission_grad(r, len(w.scene.mat_emit), g)
    # the FP64 oracle's central differences
    fd = emission_fd(osc, w.scene.mat_emit, lambda: float((gw.astype(np.float64) * oracle_means(
        osc, p, 0.0, pix, SPP, w.eps)).sum()), LIGHTS, 1e-3)
    print(ge[list(LIGHTS)], fd)
    np.testing.assert_allclose(ge[list(LIGHTS)], fd, rtol=2e-3, atol=1e-4 * np.abs(fd).max())
    assert not np.delete(ge, LIGHTS).any()
    # the same scene with its own eight materials: the same sums in FP64, up to their order
    few = sg.textured_room(seed=21, grid=40, tex_size=32)
    w.scene = few
    r8 = renderer_for(w)
    r8.set_emission(torch.from_numpy(np.asarray(few.mat_emit, np.float32)).cuda())
    np.testing.assert_allclose(ge[where], _emission_grad(r8, len(few.mat_emit), g), rtol=1e-6,
                               atol=1e-6 * np.abs(ge).max())
    r.close()
    r8.close()
