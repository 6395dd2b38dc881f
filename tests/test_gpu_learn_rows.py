"""Gradients of batches of many rows, where each CTA of the weight-gradient
kernel takes a share of 13 or more rows: its staging rings wrap, both accumulator
sets are used and a share crosses frames. Against the same frames in parts of few
rows (at most 4 rows a share, the sizes of test_gpu_learn_grads.py). The parts are
a power of two, so that dL/dz, activations and input gradients are the same bits
up to that factor and only the order of the FP32 sums over pixels differs."""
import numpy as np
import pytest

from test_gpu_learn import EPS, _features, _learned, flat, gpu_weights, rand_params, unflat

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def shifted(x):
    """x [n][c][h][w] under each tap: [9][n][c][h][w]."""
    p = torch.nn.functional.pad(x, (1, 1, 1, 1))
    h, w = x.shape[2:]
    return [p[:, :, t // 3:t // 3 + h, t % 3:t % 3 + w] for t in range(9)]


def conv(x, w):
    return sum(torch.einsum("nchw,oc->nohw", v, w[:, :, t // 3, t % 3]) for t, v in enumerate(shifted(x)))


def magnitudes(params, x, target):
    """Sum over the pixels of |dY| |X| for every weight, and of |dY| for every bias."""
    gw = [(torch.from_numpy(w).cuda(), torch.from_numpy(b).cuda()) for w, b in gpu_weights(params)]
    acts = [x]
    for w, b in gw:
        z = conv(acts[-1], w) + b[None, :, None, None]
        acts.append(z.clamp_min(0.0))
    s = torch.sigmoid(z)
    wgt = 0.05 + 0.95 * (10.0 ** (4 * x[:, :1]) - 1e-4).clamp(0, 1)
    dy = 2.0 * wgt * (EPS + (1 - EPS) * s - target[:, None]) / s.numel() * (1 - EPS) * s * (1 - s)
    out = []
    for li in range(4, -1, -1):
        o = dy.abs().transpose(0, 1).reshape(dy.shape[1], -1)
        out.append((torch.stack([o @ v.abs().transpose(0, 1).reshape(v.shape[1], -1).T for v in shifted(acts[li])], -1),
                    o.sum(1)))
        if li:
            dy = torch.where(acts[li] > 0, conv(dy, gw[li][0].flip(2, 3).transpose(0, 1)), torch.zeros_like(acts[li]))
    return out[::-1]


@pytest.mark.parametrize("ne,nz,frames,parts", [
    (16, 100, 40, 8),       # 26 rows a share, most in one frame
    (16, 1, 2000, 8),       # 13 frames of one row: three staged rows for each
    (32, 4, 704, 8),        # shares of 18 rows over five or six frames
    (64, 3, 960, 8),
    (128, 600, 4, 4),
    (128, 3, 896, 8),
])
def test_gradients_of_many_rows(ne, nz, frames, parts):
    L, _ = _learned(ne, 128, nz, max_frames=frames)
    params = rand_params(41)
    L.set_params(flat(params))
    x, feats = _features(frames, nz, ne, 42)
    tgt = torch.from_numpy(np.random.default_rng(43).uniform(EPS, 1.0, (frames, nz, ne)).astype(np.float32)).cuda()
    g, loss = L.grads(feats, tgt)
    g, loss = g.clone(), loss.clone()
    again, _ = L.grads(feats, tgt)
    assert torch.equal(g, again)
    n = frames // parts
    want, want_loss = 0.0, 0.0
    for k in range(parts):
        gk, lk = L.grads(feats[k * n:(k + 1) * n].contiguous(), tgt[k * n:(k + 1) * n].contiguous())
        want, want_loss = want + gk.double() / parts, want_loss + lk.double() / parts
    L.sync()
    L.close()
    assert abs(float(loss) - float(want_loss)) <= 1e-5 * float(want_loss)
    got, want = (unflat(v.cpu().numpy().astype(np.float64)) for v in (g, want))
    # The tensor core adds at most 4 rows' products one after the other, each rounded in FP32 at worst, then a share's
    # sums of 4 rows and 152 shares follow: 4 ne + 64 + rows / 600 roundings of 2^-24 of the terms' magnitudes, on
    # either side. The magnitudes are taken without the BF16 roundings: a few 2^-8 off, more where a channel is active
    # at a handful of pixels (1e-5 of the layer's largest for those)
    tol = 2 * 1.05 * (4 * ne + 64 + frames * nz / 600) * 2.0 ** -24
    for li, mags in enumerate(magnitudes(params, torch.from_numpy(x).cuda(), tgt.double())):
        for k in range(2):
            m = mags[k].cpu().numpy().reshape(got[li][k].shape)
            err = np.abs(got[li][k] - want[li][k])
            m = m + 1e-5 * m.max()
            assert np.all(err <= tol * m), (li, k, float(np.max(err / m)), tol)


def bf16(x):
    return x.float().bfloat16().double()


def chain(x, w):
    """s = fma(x, w, s) in FP32 over input channels, then taps."""
    xs = shifted(x)
    s = torch.zeros((x.shape[0], w.shape[0]) + x.shape[2:], dtype=torch.float64, device="cuda")
    for c in range(x.shape[1]):
        for t in range(9):
            s = (xs[t][:, None, c] * w[None, :, c, t // 3, t % 3, None, None] + s).float().double()
    return s


@pytest.mark.parametrize("ne,nz,frames", [(128, 100, 16), (64, 256, 4)])
def test_last_layers_weight_sums_round_without_bias(ne, nz, frames):
    """With targets below every prediction dL/dz is positive, as the last layer's input is: its weight gradients are
    sums of terms of one sign, where truncated additions add up. 64-bit sums of the same BF16 operands."""
    L, _ = _learned(ne, 128, nz, max_frames=frames)
    params = rand_params(45)
    L.set_params(flat(params))
    x, feats = _features(frames, nz, ne, 46)
    g, _ = L.grads(feats, torch.zeros((frames, nz, ne), device="cuda"))
    L.sync()
    got = unflat(g.cpu().numpy().astype(np.float64))[4][0]
    L.close()
    h = xt = torch.from_numpy(x).cuda()
    for li, (w, b) in enumerate(gpu_weights(params)):
        z = (chain(h, torch.from_numpy(w).cuda()) + torch.from_numpy(b).cuda()[None, :, None, None]).float().double()
        if li < 4:
            h = bf16(z.clamp_min(0.0))
    s = torch.sigmoid(z)
    wgt = 0.05 + 0.95 * (10.0 ** (4 * xt[:, :1]) - 1e-4).clamp(0, 1)
    dy = bf16(2.0 * wgt * (EPS + (1 - EPS) * s) / s.numel() * (1 - EPS) * s * (1 - s))
    o = dy.transpose(0, 1).reshape(1, -1)
    want = torch.stack([o @ v.transpose(0, 1).reshape(32, -1).T for v in shifted(h)], -1).cpu().numpy()
    err = np.linalg.norm(got.reshape(want.shape) - want) / np.linalg.norm(want)
    # A truncated step loses half an ulp, 2^-24, of a partial sum that is half its final size on average: four steps
    # 1.2e-7 (sets of 64 pixels) and eight 2.4e-7; unbiased FP32 rounding of the 152 shares and the values of dL/dz
    # that expf's last bits turn (one in 2^12 by 2^-9) add 1e-7
    assert err <= 4e-7, err
