"""How the fused kernel divides its work: the bins of few batch items over the
SMs, AS energies of several frames in groups that share a bin's phasors, and
plan launches that overlap (not while a graph is being captured). Sizes sit at
the edges of the divisions: one item, fewer bins than chunks, ragged row tiles,
a last group of one and of two frames, shares cut inside a tile and shares of
several tiles. FP64 oracle, tolerances of the plain path."""
import numpy as np
import pytest

import oracle
from gpu_common import NCC_TOL, REL_L2_TOL, rel_l2
from paper_2412_02413_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

C, PITCH, FS, Z0, DZ = 1540.0, 0.3e-3, 20e6, 4e-3, 0.45e-3


def _pam():
    from paper_2412_02413_gb300 import pam
    return pam


def _geom(ne, nt, nz, bins):
    return oracle.Geometry(ne, nt, FS, C, PITCH, nz, Z0, DZ, bins)


@pytest.mark.parametrize("ne,n_apod,frames,n_bins", [
    (16, 3, [(64, 1)], 3),                      # one item, fewer bins than chunks
    (32, 2, [(200, 130)], 11),                  # a ragged tile of DAX
    (64, 3, [(250, 50), (333, 7)], 13),         # chunks of unequal bins
    (128, 2, [(300, 33), (509, 48), (64, 1)], 17),
])
def test_batch_of_few_items(ne, n_apod, frames, n_bins):
    b = _pam().Batch(n_elem=ne, pitch=PITCH, fs=FS, c=C, frames=frames, z0=Z0, dz=DZ, n_bins=n_bins, f_lo=1e6,
                     f_hi=8e6, n_apod=n_apod, pattern_m=2)
    rfs = [synth.random_rf(ne, nt, seed=800 + i) for i, (nt, _) in enumerate(frames)]
    rf = b.pack_rf(rfs)
    img, rn = (t.clone() for t in b.as_tax(rf))
    torch.cuda.synchronize()
    b.sync()
    for i, (nt, nz) in enumerate(frames):
        orc = oracle.as_xcorr(_geom(ne, nt, nz, b.bins[i]), rfs[i], oracle.pattern(ne, n_apod, 2))
        assert rel_l2(b.unpack(img, i).cpu().numpy(), orc["image"]) <= REL_L2_TOL
        assert np.max(np.abs(b.unpack(rn, i).cpu().numpy() - orc["rho_n"])) <= NCC_TOL
    b.configure(use_graph=False, persistent_ctas=1)      # the result does not depend on the grid
    img1, rn1 = b.as_tax(rf)
    torch.cuda.synchronize()
    assert torch.equal(img1, img) and torch.equal(rn1, rn)


@pytest.mark.parametrize("ne,nt,nz,n_bins,pad", [
    (16, 64, 400, 5, False),
    (32, 128, 7, 1, False),
    (64, 128, 97, 9, False),
    (128, 256, 50, 33, False),
    (64, 256, 400, 100, False),                 # five units a CTA and more: groups on the whole chip
    (64, 128, 53, 6, True),
])
@pytest.mark.parametrize("n_frames", [2, 3, 4, 5])
def test_energies_of_several_frames(ne, nt, nz, n_bins, pad, n_frames):
    bins = list(range(4, 4 + n_bins))
    plan = _pam().Plan(n_elem=ne, pitch=PITCH, fs=FS, c=C, n_samples=nt, nz=nz, z0=Z0, dz=DZ, bins=bins, n_apod=3,
                       pattern_m=2, max_frames=n_frames, pad2x=pad)
    rf = np.stack([synth.random_rf(ne, nt, seed=850 + f) for f in range(n_frames)])
    fn = oracle.as_backprop_pad2x if pad else oracle.as_backprop
    want = [fn(_geom(ne, nt, nz, bins), rf[f]) for f in range(n_frames)]
    x = torch.from_numpy(rf).cuda()
    for grid in (0, 1, 5):
        plan.set_grid(grid)
        e = plan.as_backprop(x)
        torch.cuda.synchronize()
        plan.sync()
        for f in range(n_frames):
            assert rel_l2(e[f].cpu().numpy(), want[f]) <= REL_L2_TOL, (grid, f)


def test_captured_call_equals_the_eager_one():
    ne, nt, nz = 64, 256, 70
    plan = _pam().Plan(n_elem=ne, pitch=PITCH, fs=FS, c=C, n_samples=nt, nz=nz, z0=Z0, dz=DZ, bins=list(range(5, 45)),
                       n_apod=3, pattern_m=2, max_frames=2)
    x = torch.from_numpy(np.stack([synth.random_rf(ne, nt, seed=870 + f) for f in range(2)])).cuda()
    out = {k: v.clone() for k, v in plan.as_tax(x).items() if v is not None}
    e = plan.as_backprop(x).clone()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        got = plan.as_tax(x)
        ge = plan.as_backprop(x)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(ge, e)
    for k, v in out.items():
        assert torch.equal(got[k], v), k


@pytest.mark.parametrize("use_graph", [False, True])
def test_any_positive_grid_is_taken(use_graph):
    """A grid above the item count stands for the items' whole work, up to the
    largest number the interface takes."""
    b = _pam().Batch(n_elem=64, pitch=PITCH, fs=FS, c=C, frames=[(1024, 40)], z0=Z0, dz=DZ, n_bins=300, f_lo=1e6,
                     f_hi=8e6, n_apod=3, pattern_m=2)
    rf = b.pack_rf([synth.random_rf(64, 1024, seed=890)])
    img, rn = (t.clone() for t in b.as_tax(rf))
    for ctas in (2, 153, 2 ** 31 // 48, 2 ** 31 - 1):
        b.configure(use_graph=use_graph, persistent_ctas=ctas)
        img1, rn1 = b.as_tax(rf)
        torch.cuda.synchronize()
        assert torch.equal(img1, img) and torch.equal(rn1, rn), ctas
        assert b.info()[:2] == (1, 1)        # the grid as configure takes it: one CTA for each chunk of the one item
    b.sync()


@pytest.mark.parametrize("ne,frames,n_bins,kernels", [
    (64, [(1024, 400)] * 20, 3, 4),             # 100 items of 3 bins: dividing them costs more than it saves
    (16, [(64, 40)], 1, 4),                     # one bin cannot be divided
    (128, [(1024, 400)], 300, 5),               # 9 items of 300 bins
])
def test_items_are_divided_where_their_bins_pay_for_it(ne, frames, n_bins, kernels):
    b = _pam().Batch(n_elem=ne, pitch=PITCH, fs=FS, c=C, frames=frames, z0=Z0, dz=0.1e-3, n_bins=n_bins, f_lo=1e6,
                     f_hi=8e6, n_apod=3, pattern_m=2)
    rf = b.pack_rf([synth.random_rf(ne, nt, seed=895) for nt, _ in frames])
    img, rn = (t.clone() for t in b.as_tax(rf))
    assert b.info()[2] == kernels
    b.configure(use_graph=False, persistent_ctas=1)
    img1, rn1 = b.as_tax(rf)
    torch.cuda.synchronize()
    b.sync()
    assert torch.equal(img1, img) and torch.equal(rn1, rn)
