"""The learned form's network against a restatement of its arithmetic: every
convolution is a chain of FP32 FMAs over (input channel, tap) and activations
and gradients round to BF16, at nx = 128 (tcgen05 with the boundary cases
recomputed) as at the other widths (CUDA cores); the weight gradients are FP32
sums over the pixels in any order."""
import numpy as np
import pytest

from oracle import cnn_oracle as co
from test_gpu_learn import EPS, _features, _learned, bf16, flat, gpu_weights, rand_params, unflat

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def chain(x, w):
    """s = fma(x, w, s) in FP32 over input channels, then taps (the products of
    BF16 values are exact, so each step rounds once)."""
    n, ci, h, wd = x.shape
    xp = np.zeros((n, ci, h + 2, wd + 2))
    xp[:, :, 1:-1, 1:-1] = x
    s = np.zeros((n, w.shape[0], h, wd), np.float32)
    for c in range(ci):
        for t in range(9):
            u, v = divmod(t, 3)
            s = (xp[:, None, c, u:u + h, v:v + wd] * w[None, :, c, u, v, None, None] + s).astype(np.float32)
    return s


def forward(params, x):
    acts = [x]
    for li, (w, b) in enumerate(params):
        z = (chain(acts[-1], w) + b.astype(np.float32)[None, :, None, None]).astype(np.float32)
        if li < 4:
            acts.append(bf16(np.maximum(z, 0.0)))
    return acts, z[:, 0].astype(np.float64)


CASES = [
    (128, 1, 1),     # one output row: one CTA, a segment shorter than the staging ring
    (128, 19, 3),    # a strip of 16 rows and a ragged one; shares of the batch's rows that cross frames
    (64, 33, 2),     # four groups of 16 pixels per row
    (32, 5, 7),      # shares of several short frames
    (16, 130, 1),    # one group of 16 pixels: one split of the warps has work
]


@pytest.mark.parametrize("ne,nz,frames", CASES)
def test_network_follows_its_arithmetic(ne, nz, frames):
    L, _ = _learned(ne, 128, nz, max_frames=frames)
    params = rand_params(31)
    L.set_params(flat(params))
    x, feats = _features(frames, nz, ne, 32)
    target = np.random.default_rng(33).uniform(EPS, 1.0, (frames, nz, ne)).astype(np.float32)
    tgt = torch.from_numpy(target).cuda()
    rho = L.forward(feats).cpu().numpy()
    g, _ = L.grads(feats, tgt)
    again, _ = L.grads(feats, tgt)
    L.sync()
    assert torch.equal(g, again)
    got = unflat(g.cpu().numpy().astype(np.float64))
    gw = gpu_weights(params)
    acts, z = forward(gw, x)
    s = co.sigmoid(z)
    # the same z: rho differs by the rounding of expf, a division and a sum, a
    # few FP32 ulp; an activation rounded the other way would move it by 1e-4
    assert np.max(np.abs(rho / (EPS + (1 - EPS) * s) - 1.0)) <= 2e-6
    px = z.size
    wgt = co.loss_weights(x)[:, 0]
    dy = bf16((2.0 * wgt * (EPS + (1 - EPS) * s - target) / px * (1 - EPS) * s * (1 - s)).astype(np.float32))[:, None]
    for li in range(4, -1, -1):
        w, _ = gw[li]
        _, dw, db = co.conv3x3_backward(acts[li], w, dy)
        _, dwa, dba = co.conv3x3_backward(np.abs(acts[li]), w, np.abs(dy))
        # FP32 sum of px terms in any order: px 2^-24 of the terms' magnitudes. dL/dz
        # comes from expf: up to four of its BF16 values rounded the other way, 2^-8 each
        top = np.max(np.abs(dy)) * np.max(np.abs(acts[li]))
        slack = 4 * 2.0 ** -8 * np.array([top, np.max(np.abs(dy))])
        assert np.all(np.abs(got[li][0] - dw) <= px * 2.0 ** -24 * dwa + slack[0]), li
        assert np.all(np.abs(got[li][1] - db) <= px * 2.0 ** -24 * dba + slack[1]), li
        if li:
            dy = np.where(acts[li] > 0.0, bf16(chain(dy, np.flip(w, (2, 3)).transpose(1, 0, 2, 3))), 0.0)
    L.close()
