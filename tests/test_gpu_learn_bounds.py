"""The network's convolutions at nx = 128 (tcgen05, outputs near a BF16 rounding
boundary recomputed) and at nx = 64 (CUDA cores) where the order of the FP32 sums
shows most: a bias far larger than the sums, and terms that cancel. The layers
after the one under test pass its activations on unchanged, and the last layer
adds them up, so that rho shows every activation."""
import numpy as np
import pytest

from oracle import cnn_oracle as co
from test_gpu_learn import EPS, _features, _learned, bf16, flat, gpu_weights
from test_gpu_learn_grads import chain

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def passing(first, last):
    """Parameters with `first` in front, centre-tap identities behind it and `last` as the last layer."""
    eye = np.zeros((32, 32, 3, 3))
    eye[np.arange(32), np.arange(32), 1, 1] = 1.0
    return first + [(eye, np.zeros(32))] * (4 - len(first)) + [last]


def last_layer(seed, size, channels):
    w = np.zeros((1, 32, 3, 3))
    n = len(channels)
    w[0, channels, 1, 1] = size * np.random.default_rng(seed).uniform(0.5, 1.0, n) * (-1.0) ** np.arange(n)
    return w, np.zeros(1)


def run(ne, nz, frames, params, feats):
    L, _ = _learned(ne, 128, nz, max_frames=frames)
    L.set_params(flat(params))
    rho = L.forward(feats).cpu().numpy().astype(np.float64)
    L.sync()
    L.close()
    return rho


@pytest.mark.parametrize("ne", [64, 128])
def test_large_bias(ne):
    """A bias on a BF16 rounding boundary (1 + 2^-8) and sums around half an FP32 ulp of it: an activation is 1 or
    1 + 2^-7 by the last bits of its sum, so it shows which order made it."""
    nz, frames = 128, 16
    x, _ = _features(frames, nz, ne, 51)
    x = bf16(0.1 * x - 0.9)                     # -1 to -0.9: a narrow spread of the sums, so that many lie close by
    feats = torch.from_numpy(_pack(x)).cuda()
    w = -2.0 ** np.random.default_rng(52).uniform(-10.0, 0.0, (32, 5, 3, 3))    # of sizes whose sums have to round
    w *= 2.0 ** -24 / (0.95 * -w.sum((1, 2, 3), keepdims=True))
    params = passing([(w, np.full(32, 1 + 2.0 ** -8))], last_layer(53, 0.25, range(32)))
    gw = gpu_weights(params)
    z = (chain(x, gw[0][0]) + gw[0][1].astype(np.float32)[None, :, None, None]).astype(np.float32)
    act = bf16(z)
    assert set(np.unique(act)) == {1.0, 1.0 + 2.0 ** -7}
    zl = np.einsum("nchw,c->nhw", act, gw[4][0][0, :, 1, 1])
    want = EPS + (1 - EPS) * co.sigmoid(zl)
    rho = run(ne, nz, frames, params, feats)
    # one activation turned moves z by 2^-7 x 0.125 at least, rho by 2e-4; the rest is FP32 rounding of 32 terms and expf
    assert np.max(np.abs(rho / want - 1.0)) <= 1e-5


@pytest.mark.parametrize("layer", [0, 1])
@pytest.mark.parametrize("ne", [64, 128])
def test_cancelling_terms(ne, layer):
    """Sums whose terms cancel to a thousandth. In any order of FP32 sums the result is within n 2^-23 of the terms'
    magnitudes of the exact one (the tensor core's truncation counted), then rounds to BF16."""
    nz, frames = 33, 2
    x, _ = _features(frames, nz, ne, 61 + layer)
    x[:, 1] = x[:, 0]
    x[:, 3] = x[:, 2]
    feats = torch.from_numpy(_pack(x)).cuda()
    rng = np.random.default_rng(62)
    ci = (5, 32)[layer]
    w = np.zeros((32, ci, 3, 3))
    w[:, 0], w[:, 2] = rng.uniform(-1, 1, (2, 32, 3, 3))
    w[:, 1], w[:, 3] = -w[:, 0], -w[:, 2]
    w[:, 4] = rng.uniform(-1e-3, 1e-3, (32, 3, 3))
    first = [(w, np.zeros(32))]
    if layer:
        neg = np.zeros((32, 5, 3, 3))
        neg[np.arange(5), np.arange(5), 1, 1] = -1.0      # activations -x of the first layer
        first = [(neg, np.zeros(32))] + first
        first[1][0][:] *= -1.0
    params = passing(first, last_layer(63, 16.0, [3, 20]))
    gw = gpu_weights(params)
    h = x if layer == 0 else np.concatenate([-x, np.zeros((frames, 27, nz, ne))], 1)
    exact = np.maximum(co.conv3x3(h, gw[layer][0], np.zeros(32)), 0.0)
    size = co.conv3x3(np.abs(h), np.abs(gw[layer][0]), np.zeros(32))
    wl = gw[4][0][0, :, 1, 1]
    off = 9 * ci * 2.0 ** -23 * size + 2.0 ** -9 * exact
    off += 2.0 ** -9 * off
    zl, slack = np.einsum("nchw,c->nhw", exact, wl), np.einsum("nchw,c->nhw", off, np.abs(wl))
    rho = run(ne, nz, frames, params, feats)
    s = (rho - EPS) / (1 - EPS)
    got = np.log(s / (1 - s))
    # rho is FP32: 2^-22 of it, over the sigmoid's slope s (1 - s), and 32 FP32 additions of the last layer
    slack += 2.0 ** -22 / (s * (1 - s)) + 64 * 2.0 ** -24 * np.einsum("nchw,c->nhw", exact + off, np.abs(wl))
    assert np.all(np.abs(got - zl) <= slack), float(np.max(np.abs(got - zl) / slack))


def _pack(x):
    from paper_2412_02413_gb300 import pam
    return pam.pack_features(x)
