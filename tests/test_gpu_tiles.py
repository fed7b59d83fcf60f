"""Edges of the tiled kernels: points and rays that do not fill a tile, image sizes that do not
fill a pixel patch, every depth of the canonical MLP, odd channel counts of CNN_skel, odd widths of
the pose refiner, and volume sizes off the usual ones.

Where a kernel gives a sample the same bits wherever it lies in a launch, the tests compare launches
of different shapes bit for bit; elsewhere they compare with the FP64 oracle at the tolerances of the
other GPU tests (gradients 2e-3, transforms 2e-6, volumes 1e-4) unless a test says why not."""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import cnn
from oracle import field as OF
from oracle import refine as ORF
from oracle import render as OR
from paper_2306_16541_gb300 import synth

from _util import nrmod
from test_gpu_cnn import SMALL, _linear_subject, _oracle_volume, _prior, _rel
from test_gpu_train import _gpu_step, _oracle_grads, _setup, _smooth, u32

pytestmark = pytest.mark.gpu


def _points(n, seed=5):
    return torch.from_numpy(np.random.default_rng(seed).uniform(-0.9, 0.9, size=(n, 3)).astype(np.float32)).cuda()


@pytest.mark.parametrize("hidden", [1, 2, 3, 4])
@pytest.mark.parametrize("mlp,feat,tc", [("f32", "f32", False), ("f32", "f32", True), ("bf16", "f16", False),
                                         ("f16", "f32", False), ("fp8", "f16", False)])
def test_a_point_gives_the_same_bits_in_any_launch(hidden, mlp, feat, tc):
    """From one point (one lane of one tile, spread over the SMs) to more tiles than the chip holds."""
    nr = nrmod()
    s = synth.subject(301, hash_scale=0.5, res_last_std=0.02, hidden_layers=hidden, hash_levels=8 - hidden)
    x = _points(90001)
    S = nr.Subject(s)
    try:
        S.set_pose(*synth.random_pose(np.random.default_rng(302)))
        o = nr.make_opts(mlp, feat, f32_tc=tc)
        full = S.query(x, o).cpu().numpy()
        assert np.isfinite(full).all()
        for n in (1, 31, 32, 33, 127, 129, 1500, 20000):
            assert np.array_equal(S.query(x[:n], o).cpu().numpy(), full[:n]), n
        if hidden in (1, 4) and mlp == "f32":   # the tile layers against the oracle
            rt = np.zeros(3)
            aa, rt = synth.random_pose(np.random.default_rng(302))
            R, t, om = OR.pose_inputs(s, aa, rt)
            with torch.no_grad():
                f = OF.field(x[:500].cpu().double(), OF.Params(s), R, t, om)
            near = (f["S"] > 1e-2).numpy()      # x_skel divides by S
            assert near.sum() > 50
            ref = torch.cat([f["x_skel"], f["S"][:, None], f["x_final"], f["inside"][:, None].double(), f["rgb"],
                             f["sigma"][:, None]], 1).numpy()
            assert np.abs(full[:500] - ref)[near].max() <= 1e-3
    finally:
        S.close()


@pytest.mark.parametrize("mlp,tc", [("f32", False), ("f32", True), ("bf16", False)])
@pytest.mark.parametrize("occ,t_min", [(False, 0.0), (True, 0.0), (True, 1e-2)])
def test_a_pixel_gives_the_same_bits_in_any_image_size(mlp, tc, occ, t_min):
    """Pixel patches (40 x 24), patches over the edge (37 x 23), and rows where patches would waste
    too many rays (33 x 5, 3 x 17, 1 x 1): the same camera, so the same pixels."""
    nr = nrmod()
    s = synth.subject(303, hash_scale=0.5, res_last_std=0.02, with_ellipsoids=True)
    s["mlp_layers"][-1][1][3] = 20.0             # opaque enough for early termination
    s["mlp_params"] = synth.pack_layers(s["mlp_layers"])
    cam = synth.camera(40, 24, 30.0, (0.0, 0.0, 2.5), 150, 0.5, 4.5, bg=(0.1, 0.2, 0.3))
    S = nr.Subject(s)
    try:
        S.set_pose(*synth.random_pose(np.random.default_rng(304)))
        o = nr.make_opts(mlp, "f32", occ, t_min, f32_tc=tc)
        full = S.render(cam, o).cpu().numpy()
        assert full[..., 3].max() > 0.5
        for w, h in ((37, 23), (33, 5), (3, 17), (1, 1)):
            got = S.render(dataclasses.replace(cam, width=w, height=h), o).cpu().numpy()
            assert np.array_equal(got, full[:h, :w]), (w, h)
    finally:
        S.close()


@pytest.mark.parametrize("mlp,tc", [("f32", False), ("f32", True), ("bf16", False), ("f16", False), ("fp8", False)])
def test_samples_that_no_bone_reaches_add_nothing(mlp, tc):
    """Tiles whose samples all have S = 0 are skipped when the whole box is sampled: the image is
    that of the same samples through an occupancy grid with every cell set, which skips no tile;
    with no weights at all it is the background."""
    nr = nrmod()
    s = synth.subject(305, hash_scale=0.5, res_last_std=0.02)
    s["wvol"] = np.where(s["wvol"] > 1e-2, s["wvol"], 0.0).astype(np.float32)     # zero away from the body
    cam = synth.camera(64, 40, 40.0, (0.0, 0.0, 2.5), 96, 0.5, 4.5, bg=(0.25, 0.5, 0.75))
    pose = synth.random_pose(np.random.default_rng(306))
    for wvol in (s["wvol"], np.zeros_like(s["wvol"])):
        S = nr.Subject(dict(s, wvol=wvol))
        try:
            S.set_pose(*pose)
            S.set_canonical_occupancy(np.full(128 ** 3 // 32, 0xFFFFFFFF, np.uint32), 0.0)
            assert (S.occupancy() == 0xFFFFFFFF).all()
            for t_min in (0.0, 1e-4):
                a, b = (S.render(cam, nr.make_opts(mlp, "f16", occ, t_min, f32_tc=tc)).cpu().numpy()
                        for occ in (False, True))
                assert np.array_equal(a, b)
        finally:
            S.close()
        if wvol.any():
            assert a[..., 3].max() > 0.05
        else:
            assert (a == np.array([0.25, 0.5, 0.75, 0.0], np.float32)).all()


@pytest.mark.parametrize("S,n_rays,hidden", [(1, 70, 2), (7, 150, 3), (48, 90, 2), (100, 37, 4), (200, 20, 1),
                                             (600, 9, 2)])
def test_gradients_match_oracle_at_ray_lengths_off_the_tile(S, n_rays, hidden):
    """Rays that straddle warps, groups that do not fill a block, more samples than a block holds
    (the separate forward and compositing kernels), every MLP depth; few samples, so that the weight
    volume's gradient is scattered without the corner-block sums -- and so that one sample on the
    other side of a kink weighs up to a few parts in a thousand: 1e-2."""
    _, frames, batch, tgt = _setup(n_rays=n_rays, S=S, seed=311)
    subj = _smooth(synth.subject(311, hash_scale=0.5, res_last_std=0.02, hidden_layers=hidden))
    loss, g, _, _ = _gpu_step(subj, frames, batch, tgt, S, 7, True)
    ref_loss, ref = _oracle_grads(subj, frames, batch, tgt, S, 7)
    assert abs(loss - ref_loss) <= 1e-5 * max(1.0, ref_loss)
    for k in ("table", "mlp", "res"):
        assert _rel(g[k], ref[k]) <= 1e-2, (k, _rel(g[k], ref[k]))
    assert np.isfinite(g["wvol"]).all() and np.linalg.norm(g["wvol"]) > 0


@pytest.mark.parametrize("vol_res", [2, 17, 33])
def test_corner_block_sums_equal_the_direct_scatter(vol_res):
    """The same rays once in a batch small enough for the direct scatter and once in one large enough
    for the corner-block sums (the first rays with a loss, the rest without): rays keep their index,
    so they keep their samples."""
    nr = nrmod()
    s = synth.subject(313, vol_res=vol_res, hash_scale=0.5, res_last_std=0.02)
    frames = synth.training_frames(314, 3, res=64)
    n, S = 24, 32
    quad = (vol_res + 2) * (vol_res + 1) ** 2 * 24 * 16
    assert quad > 512 * n * S or vol_res == 2
    many = max(n, -(-quad // (512 * S)) + 1)
    b = synth.pixel_batch(315, many, 3, 64, 64)
    grads = []
    for m in (n, many):
        sub = nr.Subject(s)
        try:
            sub.set_frames(frames["axis_angle"], frames["root_t"], frames["cameras"])
            g = torch.zeros(m, 3, device="cuda")
            g[:n] = torch.linspace(-1, 1, 3 * n, device="cuda").reshape(n, 3)
            sub.train_step(u32(b["frame"][:m]), u32(b["px"][:m]), u32(b["py"][:m]), None, S, 3, grad_rgb=g, grad_only=True)
            grads.append(sub.param(nr.NR_PARAM_WVOL)[1].cpu().numpy().astype(np.float64))
        finally:
            sub.close()
    assert np.linalg.norm(grads[0]) > 0
    assert _rel(grads[1], grads[0]) <= 1e-5


@pytest.mark.parametrize("vol_res", [2, 33, 70])
def test_support_boxes_drop_only_negligible_weights(vol_res):
    """The boxes hold every vertex above 1e-7, so S moves by at most 24 x 1e-7 (and rounding)."""
    nr = nrmod()
    s = synth.subject(317, vol_res=vol_res)
    x = _points(20000, 318)
    S = nr.Subject(s)
    try:
        S.set_pose(*synth.random_pose(np.random.default_rng(319)))
        a = S.query(x, nr.make_opts("f32")).cpu().numpy()[:, 3]
        b = S.query(x, nr.make_opts("f32", all_bones=True)).cpu().numpy()[:, 3]
    finally:
        S.close()
    assert np.abs(a - b).max() <= 2.4e-6 + 24 * 2.0 ** -24 * max(1.0, b.max())


@pytest.mark.parametrize("channels", [(3, 5, 7, 6, 9), (40, 24, 18, 20, 17), (1, 1, 1, 1, 1)])
def test_generator_with_odd_channel_counts(channels):
    """Channel counts off every tile (and off 16-byte alignment): the volume, and the gradient of a
    training step in every weight."""
    nr = nrmod()
    subj = _linear_subject(321)
    layers = synth.cnn_layers(322, channels, last_std=0.3)
    z, prior = synth.cnn_latent(323), _prior(synth.subject(321))
    frames = synth.training_frames(324, 2, res=32)
    for c in frames["cameras"]:
        c.n_samples = 16
    batch = synth.pixel_batch(325, 300, 2, 32, 32)
    tgt = np.random.default_rng(326).uniform(0, 1, size=(300, 3)).astype(np.float32)
    sub = nr.Subject(subj)
    try:
        sub.set_weight_cnn(layers, z, prior)
        sub.set_frames(frames["axis_angle"], frames["root_t"], frames["cameras"])
        sub.train_step(u32(batch["frame"]), u32(batch["px"]), u32(batch["py"]), torch.from_numpy(tgt).cuda(), 16, 5,
                       grad_only=True)
        grad = sub.param(nr.NR_PARAM_CNN)[1].cpu().numpy().astype(np.float64)
        vol = sub.param(nr.NR_PARAM_WVOL)[0].cpu().numpy().reshape(25, 32, 32, 32)
    finally:
        sub.close()
    ref_vol = _oracle_volume(layers, z, prior)
    assert np.abs(vol - ref_vol).max() <= 1e-5 + 1e-4 * np.abs(ref_vol).max()
    L = cnn.as_tensors(layers, requires_grad=True)
    P = OF.Params(subj)
    P.wvol = cnn.weight_volume(L, torch.from_numpy(z.astype(np.float64)), torch.from_numpy(prior.astype(np.float64)))
    OR.train_loss(subj, P, frames, batch, tgt, 5, 16, np.zeros(3))[0].backward()
    ref = np.concatenate([np.concatenate([W.grad.numpy().ravel(), b.grad.numpy().ravel()]) for W, b in L])
    assert _rel(grad, ref) <= 2e-3, _rel(grad, ref)


@pytest.mark.parametrize("width,hidden", [(1, 1), (17, 3), (100, 4), (255, 2)])
def test_refiner_widths_off_the_tile(width, hidden):
    nr = nrmod()
    s = synth.subject(331)
    layers = synth.refiner_layers(332, width, hidden, 0.05)
    aa, rt = synth.random_pose(np.random.default_rng(333))
    S = nr.Subject(s)
    try:
        S.set_pose_refiner(layers)
        S.set_pose(aa, rt)
        G = S.pose_transforms()
    finally:
        S.close()
    t64 = [(torch.from_numpy(W.astype(np.float64)), torch.from_numpy(b.astype(np.float64))) for W, b in layers]
    R, t = ORF.refined_transforms(s["parents"], s["rest_joints"], aa, rt, t64)
    ref = np.concatenate([R.numpy(), t.numpy()[:, :, None]], 2).reshape(-1, 12)
    assert np.abs(G - ref).max() <= 2e-6
