"""Forms that other tests leave out: float32 renders against a reference that skips nothing, the
weight volume's gradient on both of its routes and at ray lengths off the tile, boxes whose cells are
no powers of two, and static renders whose size is no whole number of pixel patches."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2306_16541_gb300 import synth

from _util import nrmod, oracle_render
from test_gpu_cnn import _linear_subject, _rel
from test_gpu_train import _gpu_step, _oracle_grads, _setup, u32

pytestmark = pytest.mark.gpu

TOL = 1e-3      # the float32 tolerance of the parity tests


@pytest.mark.parametrize("tc", [False, True])
def test_float32_tiles_left_out_add_nothing(tc):
    """The float32 kernels skip a tile whose samples all have S = 0 in every render, so the reference
    is the oracle, which evaluates each sample: the volume is zero away from the body."""
    nr = nrmod()
    s = synth.subject(441, hash_scale=0.5, res_last_std=0.02)
    s["wvol"] = np.where(s["wvol"] > 1e-2, s["wvol"], 0.0).astype(np.float32)
    cam = synth.camera(40, 24, 25.0, (0.0, 0.0, 2.5), 40, 0.5, 4.5, bg=(0.25, 0.5, 0.75))
    pose = synth.random_pose(np.random.default_rng(442))
    ref = oracle_render(s, pose, cam, False).reshape(24, 40, 4)
    assert ref[..., 3].max() > 0.05 and (ref[..., 3] == 0).mean() > 0.2
    S = nr.Subject(s)
    try:
        S.set_pose(*pose)
        img = S.render(cam, nr.make_opts("f32", f32_tc=tc)).cpu().numpy()
    finally:
        S.close()
    assert np.abs(img - ref).max() <= TOL


def test_smallest_volume_gradient_on_both_routes():
    """A 2^3 volume: one ray of 16 samples scatters directly (the corner blocks' 13,824 bytes are more
    than 512 a sample), two go through the corner-block sums, the second without a gradient."""
    nr = nrmod()
    s = synth.subject(443, vol_res=2, hash_scale=0.5, res_last_std=0.02)
    frames = synth.training_frames(444, 1, res=64)
    grads = []
    for n in (1, 2):
        assert (4 * 3 ** 2 * 24 * 16 > 512 * 16 * n) == (n == 1)
        sub = nr.Subject(s)
        try:
            sub.set_frames(frames["axis_angle"], frames["root_t"], frames["cameras"])
            g = torch.tensor([[0.3, -0.2, 0.5], [0.0, 0.0, 0.0]], device="cuda")[:n].contiguous()
            sub.train_step(u32(np.zeros(n)), u32(np.full(n, 32)), u32(np.full(n, 32)), None, 16, 3, grad_rgb=g,
                           grad_only=True)
            grads.append(sub.param(nr.NR_PARAM_WVOL)[1].cpu().numpy().astype(np.float64))
        finally:
            sub.close()
    assert np.linalg.norm(grads[0]) > 0
    assert _rel(grads[1], grads[0]) <= 1e-5


@pytest.mark.parametrize("S,n_rays", [(7, 300), (48, 90), (200, 30), (600, 12)])
def test_volume_gradient_matches_oracle_at_ray_lengths_off_the_tile(S, n_rays):
    """A field that is linear in space on two coarse levels, so that no hash cell's face makes a kink;
    1e-2 as for the other groups of the same batches."""
    subj = _linear_subject(445)
    _, frames, batch, tgt = _setup(n_rays=n_rays, S=S, seed=446)
    loss, g, _, _ = _gpu_step(subj, frames, batch, tgt, S, 7, True)
    ref_loss, ref = _oracle_grads(subj, frames, batch, tgt, S, 7)
    assert abs(loss - ref_loss) <= 1e-5 * max(1.0, ref_loss)
    assert _rel(g["wvol"], ref["wvol"]) <= 1e-2, _rel(g["wvol"], ref["wvol"])


def _odd_box(seed):
    s = synth.subject(seed, hash_scale=0.5, res_last_std=0.02, with_ellipsoids=True)
    s["box_min"] = np.array([-1.05, -1.1, -1.0], np.float32)
    s["box_max"] = np.array([1.1, 1.05, 1.07], np.float32)
    return s


@pytest.mark.parametrize("occ", [False, True])
def test_a_box_whose_cells_are_no_powers_of_two(occ):
    nr = nrmod()
    s = _odd_box(447)
    cam = synth.camera(37, 23, 25.0, (0.0, 0.0, 2.5), 40, 0.5, 4.5, bg=(0.1, 0.2, 0.3))
    pose = synth.random_pose(np.random.default_rng(448))
    ref = oracle_render(s, pose, cam, occ).reshape(23, 37, 4)
    assert ref[..., 3].max() > 0.05
    S = nr.Subject(s)
    try:
        S.set_pose(*pose)
        img = S.render(cam, nr.make_opts("f32", occupancy=occ)).cpu().numpy()
    finally:
        S.close()
    assert np.abs(img - ref).max() <= TOL


@pytest.mark.parametrize("odd", [False, True])
@pytest.mark.parametrize("w,h", [(61, 63), (40, 23), (33, 5), (7, 4), (1, 1)])
def test_static_renders_off_the_patch(w, h, odd):
    """In row order where the patches do not cover the image exactly: the pixels of nr_render."""
    nr = nrmod()
    s = _odd_box(449) if odd else synth.subject(449, hash_scale=0.5, res_last_std=0.02, with_ellipsoids=True)
    cam = nr.make_camera(dataclasses.replace(synth.camera(64, 64, 50.0, (0.0, 0.0, 2.5), 60, 0.5, 4.5), width=w, height=h))
    S = nr.Subject(s)
    try:
        S.set_pose(*synth.random_pose(np.random.default_rng(450)))
        for mlp, occ, t_min in (("f32", True, 0.0), ("bf16", True, 1e-3), ("bf16", False, 0.0)):
            o = nr.make_opts(mlp, "f32" if mlp == "f32" else "f16", occ, t_min)
            out = torch.full((h, w, 4), float("nan"), device="cuda")
            nr.nr_render_static(S.h, cam, o, out)
            assert torch.equal(out, S.render(cam, o)), (mlp, occ, t_min)
    finally:
        S.close()
