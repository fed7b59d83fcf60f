"""Values that are not finite: a NaN or an infinity that enters a training step or a weight must
reach everything that depends on it, so that a caller who looks at any gradient sees it."""
import numpy as np
import pytest
import torch

from paper_2306_16541_gb300 import synth

from _util import nrmod
from test_gpu_cnn import SMALL, _prior
from test_gpu_train import u32

pytestmark = pytest.mark.gpu

CUDA_NAN = 0x7FFFFFFF      # the NaN that GPU arithmetic produces (a stored one may have other bits)


def _matrices(flat, layers):
    """The weight matrices of a packed group (W then b of each layer)."""
    out, o = [], 0
    for W, b in layers:
        out.append(flat[o:o + W.size])
        o += W.size + b.size
    return out


@pytest.mark.parametrize("value", [float("nan"), float("inf"), float("-inf")])
@pytest.mark.parametrize("S,hidden", [(32, 2), (48, 4), (600, 1)])
def test_a_bad_loss_gradient_reaches_every_group(value, S, hidden):
    """dL/dC of one ray in the batch, in the fused step (32, 48 samples) and in the separate kernels
    (600): the weights of every layer, not only of the last, and the hash table, the volume's
    generator and the pose refiner."""
    nr = nrmod()
    s = synth.subject(401, hash_scale=0.5, res_last_std=0.02, hidden_layers=hidden)
    frames = synth.training_frames(402, 1, res=32)
    sub = nr.Subject(s)
    try:
        sub.set_weight_cnn(synth.cnn_layers(403, SMALL, last_std=0.3), synth.cnn_latent(404), _prior(s))
        sub.set_pose_refiner(synth.refiner_layers(405, 32, 1, 0.05))
        sub.set_frames(frames["axis_angle"], frames["root_t"], frames["cameras"])
        n = 16
        fr, px, py = (u32(a) for a in (np.zeros(n), np.full(n, 15), np.arange(8, 8 + n)))   # through the body
        g = torch.full((n, 3), 0.1, device="cuda")
        for bad in (False, True):
            if bad:
                g[7] = value
            sub.train_step(fr, px, py, None, S, 3, grad_rgb=g, grad_only=True)
            mlp, res = (sub.param(k)[1].cpu().numpy() for k in (nr.NR_PARAM_MLP, nr.NR_PARAM_RES))
            groups = {f"mlp {i}": w for i, w in enumerate(_matrices(mlp, s["mlp_layers"]))}
            groups.update({f"res {i}": w for i, w in enumerate(_matrices(res, s["res_layers"]))})
            for k in ("WVOL", "HASH", "REFINER", "CNN"):
                groups[k] = sub.param(getattr(nr, "NR_PARAM_" + k))[1].cpu().numpy()
            for k, v in groups.items():
                assert np.isfinite(v).all() != bad, k
                assert np.any(v != 0), k
    finally:
        sub.close()


@pytest.mark.parametrize("bits", [CUDA_NAN, 0x7FC00000, 0x7F800001, 0xFFFFFFFF, 0x7F800000])
@pytest.mark.parametrize("tc", [False, True])
def test_a_bad_output_weight_shows(bits, tc):
    """A weight of the density's row that is not finite: no density of a query or a pixel is finite
    where the layer's input is not zero, in either float32 tier and in the training forward."""
    nr = nrmod()
    s = synth.subject(411, hash_scale=0.5, res_last_std=0.02)
    s["mlp_layers"][-2][1][5] = 10.0             # unit 5 of the last hidden layer is always on
    s["mlp_params"] = synth.pack_layers(s["mlp_layers"])
    x = torch.from_numpy(np.random.default_rng(412).uniform(-0.5, 0.5, (100, 3)).astype(np.float32)).cuda()
    frames = synth.training_frames(413, 1, res=32)
    sub = nr.Subject(s)
    try:
        sub.set_pose(frames["axis_angle"][0], frames["root_t"][0])
        sub.set_frames(frames["axis_angle"], frames["root_t"], frames["cameras"])
        W, b = s["mlp_layers"][-1]
        p = sub.param(nr.NR_PARAM_MLP)[0]
        p.view(torch.int32)[-(W.size + b.size) + 3 * 64 + 5] = int(np.uint32(bits).view(np.int32))
        sub.params_changed()
        torch.cuda.synchronize()
        o = nr.make_opts("f32", f32_tc=tc)
        sigma = sub.query(x, o)[:, 11].cpu().numpy()
        assert not np.isfinite(sigma).any()
        if bits != 0x7F800000:                   # (an infinite density is an opaque pixel)
            img = sub.render(frames["cameras"][0], o)[15, 12:20].cpu().numpy()
            assert not np.isfinite(img).any()
            pred = torch.zeros(8, 3, device="cuda")
            loss = sub.train_step(u32(np.zeros(8)), u32(np.arange(12, 20)), u32(np.full(8, 15)), torch.zeros_like(pred),
                                  32, 3, pred_rgb=pred, grad_only=True)
            assert not np.isfinite(loss) and not torch.isfinite(pred).any()
    finally:
        sub.close()


def test_a_bad_weight_of_a_tap_that_reaches_nothing_stays_alone():
    """The generator's first transposed convolution takes one voxel to 2^3: the outer taps of its 4^3
    kernels reach nothing, so their values enter neither the volume nor any gradient."""
    nr = nrmod()
    s = synth.subject(421)
    layers = synth.cnn_layers(422, SMALL, last_std=0.3)
    frames = synth.training_frames(423, 1, res=32)
    sub = nr.Subject(s)
    try:
        sub.set_weight_cnn(layers, synth.cnn_latent(424), _prior(s))
        sub.set_frames(frames["axis_angle"], frames["root_t"], frames["cameras"])
        n = 16
        rays = [u32(a) for a in (np.zeros(n), np.full(n, 15), np.arange(8, 8 + n))]
        p, g = sub.param(nr.NR_PARAM_CNN)
        o = layers[0][0].size + layers[0][1].size
        W1 = p[o:o + layers[1][0].size].view(*layers[1][0].shape)
        grads = []
        for bad in (False, True):
            if bad:
                W1[2, 3, 0, 1, 2] = float("inf")
                W1[5, 7, 2, 3, 1] = float("nan")
                sub.params_changed()
            sub.train_step(*rays, None, 32, 3, grad_rgb=torch.full((n, 3), 0.1, device="cuda"), grad_only=True)
            assert torch.isfinite(sub.param(nr.NR_PARAM_WVOL)[0]).all()
            grads.append(g.cpu().numpy())
    finally:
        sub.close()
    assert np.isfinite(grads[1]).all() and np.any(grads[0] != 0)
    assert np.linalg.norm(grads[1] - grads[0]) <= 1e-4 * np.linalg.norm(grads[0])   # (sums by atomics)
