"""The workloads this library's speed is measured on, with their inputs and exact values.

Each case is one call a user's program makes: a single frame as it arrives, a
block of recorded frames, a host-to-host call, an uneven batch, a tensor-core
form, a gradient of the learned form or its inference. Channel data are
synthetic frames of point sources (harmonic and broadband emissions, 1/r
spreading, 20 dB noise), as in ``paper_2412_02413_gb300.synth`` but generated
on the GPU. ``exact`` restates the method in 64 bits with torch alone.
"""
import math

import numpy as np
import torch

from paper_2412_02413_gb300 import learn, pam

C = 1540.0          # m/s
PITCH = 0.3e-3      # m
EPS = 1e-3          # NCC floor
DZ = 55e-3 / 511    # depth step of the 128 x 512 grid over 5-60 mm
FEATURE_FLOOR = 1e-4
WEIGHT_FLOOR = 0.05


def listed():
    wide = dict(ne=128, nt=4096, fs=40e6, nz=512, n_bins=300, f_lo=0.5e6, f_hi=8e6, z0=5e-3, dz=DZ, pattern=16)
    mid = dict(ne=64, nt=1024, fs=20e6, nz=128, n_bins=307, f_lo=1e6, f_hi=7e6, z0=10e-3, dz=40e-3 / 127, pattern=8)
    return [
        # live imaging on the 128-element array: one frame per call, image and NCC weight shown
        dict(wide, name="frame_128", kind="tax", frames=1),
        # offline processing of a recording: 64 frames per call
        dict(wide, name="frames_128_x64", kind="tax", frames=64),
        # acquisition on the host, 64-element array: pinned buffers in and out, the call blocks until the map is there
        dict(mid, name="host_64", kind="host", frames=1),
        # the smallest calls: a 16-element strip previewed over a few depths, where launches count
        dict(name="preview_16", kind="tax", ne=16, nt=128, fs=20e6, nz=7, n_bins=45, f_lo=1e6, f_hi=8e6, z0=4e-3,
             dz=0.45e-3, pattern=2, frames=1),
        # two complementary apertures on a small array, evanescent components dropped, every map kept, ragged rows
        dict(name="dax_32_x5", kind="dax", ne=32, nt=256, fs=20e6, nz=77, n_bins=20, f_lo=1e6, f_hi=8e6, z0=4e-3,
             dz=0.45e-3, pattern=4, frames=5, evanescent_zero=True, all_maps=True),
        # plain angular-spectrum energy (no apodization), the comparison image, odd depth count
        dict(name="energy_128_x7", kind="as", ne=128, nt=2048, fs=40e6, nz=301, n_bins=200, f_lo=0.5e6, f_hi=8e6,
             z0=5e-3, dz=DZ, pattern=16, frames=7),
        # lateral padding against wrap-around on the 64-element array, with the pair NCCs and the AS map
        dict(mid, name="padded_64_x3", kind="tax", frames=3, pad2x=True, all_maps=True),
        # high-throughput processing at FP32-level accuracy on the tensor cores
        dict(wide, name="fp16split_128_x64", kind="tax", frames=64, form="fp16split"),
        # fast overview at 16-bit accuracy, a frame count that fills no group
        dict(wide, name="bf16_128_x21", kind="tax", frames=21, form="bf16"),
        # recordings of different lengths and depth ranges in one call
        dict(name="uneven_128_x64", kind="batch", ne=128, fs=40e6, n_bins=300, f_lo=0.5e6, f_hi=8e6, z0=5e-3, dz=DZ,
             pattern=16, frames=64, nt_lo=1024, nt_hi=8192, nz_lo=128, nz_hi=512),
        # one gradient of the learned weight at the training's batch size (forward, loss, backward)
        dict(name="gradients_128_x16", kind="grads", ne=128, nz=512, frames=16),
        # learned imaging with the error gate and its fallback
        dict(wide, name="learned_128_x32", kind="learned", frames=32, gate=0.25),
    ]


def _cost(c):
    """Propagation work of a case in units of (bin, row, frame), scaled to the 128-point transform."""
    nz = 0.5 * (c["nz_lo"] + c["nz_hi"]) if c["kind"] == "batch" else c["nz"]
    nx = c["ne"] * (2 if c.get("pad2x") or c.get("upsample2x") else 1)
    return nz * c["frames"] * c.get("n_bins", 300) * nx / 128


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    while True:
        kind = rng.choice(["tax", "tax", "tax", "dax", "as", "host", "form", "form", "batch", "grads", "learned"])
        c = dict(kind=kind, frames=log_int(1, 64))
        if kind == "grads":
            c.update(ne=rng.choice([64, 128, 128]), nz=log_int(48, 512), frames=log_int(1, 16))
            return c
        wide = kind in ("form", "learned") or rng.random() < 0.5
        c.update(ne=128 if wide else rng.choice([16, 32, 64]), fs=rng.choice([20e6, 40e6]), f_lo=rng.choice([0.5e6, 1e6]),
                 f_hi=rng.uniform(5e6, 8e6), z0=rng.uniform(4e-3, 10e-3), dz=rng.uniform(0.08e-3, 0.45e-3))
        c.update(pattern=c["ne"] // 8, n_bins=log_int(20, 400))
        if kind == "batch":
            nt, nz = log_int(600, 3000), log_int(30, 256)
            c.update(nt_lo=nt, nt_hi=nt + rng.randint(1, 5000), nz_lo=nz, nz_hi=nz + rng.randint(1, 256))
        else:
            c.update(nt=2 ** rng.randint(9, 12) if kind == "learned" else 2 ** rng.randint(7, 13), nz=log_int(7, 700))
        if kind == "form":
            c.update(kind="tax", form=rng.choice(["bf16", "fp16", "fp16split", "bf16split"]))
        if kind == "learned":
            c.update(gate=rng.choice([0.1, 0.25, 0.5]), n_bins=max(40, c["n_bins"]))
        if kind in ("tax", "dax"):
            c.update(all_maps=rng.random() < 0.4, evanescent_zero=rng.random() < 0.3)
            if c["ne"] <= 64 and rng.random() < 0.4:
                c[rng.choice(["pad2x", "upsample2x"])] = True
        if _cost(c) <= 300 * 512 * 64:
            return c


# ------------------------------------------------------------------ inputs --
def _bins(c, nt=None):
    """n_bins of the band's bins spread evenly (all of them where the band holds fewer)."""
    nt = c["nt"] if nt is None else nt
    df = c["fs"] / nt
    lo = max(1, math.ceil(c["f_lo"] / df - 1e-9))
    hi = min((nt - 1) // 2, math.floor(c["f_hi"] / df + 1e-9))
    k, n = hi - lo + 1, c["n_bins"]
    if n >= k:
        return np.arange(lo, hi + 1)
    i = np.arange(n)
    return lo + (2 * i * (k - 1) + n - 1) // (2 * (n - 1))


def _uneven(c):
    """(n_samples, nz) of each frame of an uneven batch: a property of the recordings, not of the seed."""
    rng = np.random.default_rng([c["frames"], c["nt_lo"], c["nz_lo"]])
    return [(int(rng.integers(c["nt_lo"], c["nt_hi"] + 1)), int(rng.integers(c["nz_lo"], c["nz_hi"] + 1)))
            for _ in range(c["frames"])]


def _frame(c, nt, nz, rng, gen):
    """Channel data [ne][nt] of 1-6 point sources inside the imaged region."""
    ne, fs = c["ne"], c["fs"]
    dev = "cuda"
    xe = (torch.arange(ne, device=dev, dtype=torch.float64) - (ne - 1) / 2) * PITCH
    t = torch.arange(nt, device=dev, dtype=torch.float64) / fs
    fl = torch.fft.rfftfreq(2 * nt, 1 / fs, device=dev, dtype=torch.float64)
    band = ((fl >= 0.8 * c["f_lo"]) & (fl <= 1.05 * c["f_hi"])).double()
    rf = torch.zeros((ne, nt), device=dev, dtype=torch.float64)
    spec = torch.zeros((ne, nt + 1), device=dev, dtype=torch.complex128)
    for s in range(int(rng.integers(1, 7))):
        x = (rng.uniform(0.06, 0.94) - 0.5) * (ne - 1) * PITCH
        z = c["z0"] + rng.uniform(0.1, 0.9) * max(nz - 1, 1) * c["dz"]
        f0, amp, stable = float(rng.choice([1.0e6, 1.5e6])), rng.uniform(0.5, 1.0), s % 2 == 0
        r = torch.sqrt((xe - x) ** 2 + z * z)
        gain = 10e-3 / r
        if stable:
            h = np.arange(2, 2 * int(min(fs / 2, 1.05 * c["f_hi"]) / f0) + 1) / 2     # harmonics and ultra-harmonics
            f = torch.from_numpy(h * f0).to(dev)
            a = torch.from_numpy(amp * np.where(h % 1 == 0, 1.0, 0.3) / np.sqrt(np.floor(h))).to(dev)
            ph = torch.from_numpy(rng.uniform(0, 2 * np.pi, h.size)).to(dev)
            at = ph[None] - 2 * np.pi * f[None] * (r / C)[:, None]
            wt = 2 * np.pi * f[:, None] * t[None]
            rf += gain[:, None] * ((torch.cos(at) * a) @ torch.sin(wt) + (torch.sin(at) * a) @ torch.cos(wt))
        q = torch.complex(*torch.randn((2, nt + 1), generator=gen, device=dev, dtype=torch.float64)) * band
        q *= (0.1 if stable else 1.0) * amp / torch.fft.irfft(q, 2 * nt).std().clamp_min(1e-12)
        tau = torch.polar(gain[:, None].expand(ne, nt + 1).contiguous(), -2 * np.pi * (r / C)[:, None] * fl[None])
        spec += q[None] * tau
    rf += torch.fft.irfft(spec, 2 * nt)[:, :nt]
    noise = torch.randn((ne, nt), generator=gen, device=dev, dtype=torch.float64)
    return (rf + noise * rf.pow(2).mean().sqrt() * 10 ** (-20 / 20)).float()


def _frames(c, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.default_rng(seed)
    if c["kind"] == "batch":
        return [_frame(c, nt, nz, rng, gen) for nt, nz in _uneven(c)]
    return torch.stack([_frame(c, c["nt"], c["nz"], rng, gen) for _ in range(c["frames"])])


def _training_batch(c, seed):
    """Packed network inputs (BF16 [n][nz+2][nx+2][8]) and target weights of
    synthetic energy maps: a few bright spots over a speckled background."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n, nz, nx = c["frames"], c["nz"], c["ne"]

    def uniform(*shape):
        return torch.rand(shape, generator=gen, device="cuda")

    j = torch.arange(nz, device="cuda").view(1, 1, nz, 1)
    i = torch.arange(nx, device="cuda").view(1, 1, 1, nx)
    spots = torch.zeros((n, 1, nz, nx), device="cuda")
    for _ in range(4):
        pz, px, s, a = uniform(n, 1, 1, 1) * nz, uniform(n, 1, 1, 1) * nx, 1 + 3 * uniform(n, 1, 1, 1), uniform(n, 1, 1, 1)
        spots = spots + a * torch.exp(-((j - pz) / (3 * s)) ** 2 - ((i - px) / s) ** 2)
    bands = (spots + 0.02) * (0.2 - torch.log(uniform(n, 4, nz, nx).clamp_min(1e-6)))
    e = bands.sum(1, keepdim=True)
    x = torch.log10(torch.cat([e, bands], 1) / e.amax((1, 2, 3), keepdim=True) + FEATURE_FLOOR) / 4
    feats = torch.zeros((n, nz + 2, nx + 2, 8), dtype=torch.bfloat16, device="cuda")
    feats[:, 1:-1, 1:-1, :5] = x.permute(0, 2, 3, 1).bfloat16()
    target = (EPS + (1 - EPS) * (spots / (spots + 0.2)) * (0.7 + 0.3 * uniform(n, 1, nz, nx)))[:, 0].contiguous()
    return feats.view(torch.uint8).view(n, -1), target


# ------------------------------------------------------------------- calls --
def _geometry(c):
    return dict(n_elem=c["ne"], pitch=PITCH, fs=c["fs"], c=C, n_samples=c["nt"], nz=c["nz"], z0=c["z0"], dz=c["dz"],
                bins=_bins(c), pattern_m=c["pattern"], max_frames=c["frames"])


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"case": c}
    if kind == "grads":
        s["features"], s["target"] = _training_batch(c, seed)
        s["net"] = pam.Learned(c["ne"], PITCH, 40e6, C, 256, c["nz"], 5e-3, DZ, bins=range(4, 52),
                               max_frames=c["frames"])
        s["net"].set_params(learn.load_checkpoint()[0])
        return s
    rf = _frames(c, seed)
    if kind == "batch":
        b = s["batch"] = pam.Batch(c["ne"], PITCH, c["fs"], C, _uneven(c), c["z0"], c["dz"], c["n_bins"], c["f_lo"],
                                   c["f_hi"], pattern_m=c["pattern"])
        s["rf"] = torch.zeros(b.rf_total, device="cuda")
        for f, at in zip(rf, b.rf_offsets):
            s["rf"][at:at + f.numel()] = f.reshape(-1)
        s["image"], s["rho_n"] = torch.empty((2, (b.map_total + 3) // 4 * 4), device="cuda")
        return s
    if kind == "learned":
        s["net"] = pam.Learned(**_geometry(c))
        s["net"].set_params(learn.load_checkpoint()[0])
        s["net"].configure(gate_tol=c["gate"], tensor_cores=True)
    else:
        s["plan"] = pam.Plan(n_apod={"as": 1, "dax": 2}.get(kind, 3), form=c.get("form", "fp32"),
                             evanescent_zero=c.get("evanescent_zero", False), pad2x=c.get("pad2x", False),
                             upsample2x=c.get("upsample2x", False), **_geometry(c))
    s["rf"] = rf
    if kind == "host":
        s["rf"] = rf.cpu().pin_memory().numpy()
        s["image"], s["rho_n"] = (torch.empty((c["frames"], c["nz"], c["ne"]), pin_memory=True).numpy() for _ in "ab")
    return s


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "grads":
        grads, loss = state["net"].grads(state["features"], state["target"])
        return {"grads": grads, "loss": loss}
    if kind == "batch":
        image, rho_n = state["batch"].as_tax(state["rf"], image=state["image"], rho_n=state["rho_n"])
        n = state["batch"].map_total
        return {"image": image[:n], "rho_n": rho_n[:n]}
    if kind == "host":
        state["plan"].as_xcorr_host(state["rf"], state["image"], state["rho_n"])
        return {"image": state["image"], "rho_n": state["rho_n"]}
    if kind == "learned":
        return state["net"].as_tax(state["rf"])
    if kind == "as":
        return {"energy": state["plan"].as_backprop(state["rf"])}
    call = state["plan"].as_dax if kind == "dax" else state["plan"].as_tax
    return call(state["rf"], rho_pairs=c.get("all_maps", False), image_as=c.get("all_maps", False))


def _map_flops(ne, nt, nz, n_bins, nx, apertures):
    """A real FFT per channel, the lateral FFTs, and per (bin, row) a phase and
    an inverse FFT per aperture and the correlation sums."""
    sums = {1: 1, 2: 3, 3: 6}[apertures]
    lateral = 5 * nx * math.log2(nx)
    return 2.5 * ne * nt * math.log2(nt) + n_bins * apertures * lateral + \
        n_bins * nz * (apertures * (6 * nx + lateral) + 4 * sums * nx)


def work(case):
    c, kind, n = case, case["kind"], case["frames"]
    if kind == "grads":
        px = n * c["nz"] * c["ne"]
        macs = 9 * (5 * 32 + 3 * 32 * 32 + 32)
        return {"bytes": px * (8 * 2 + 4) + 4 * 29505, "flops": px * (6.0 * macs - 2 * 9 * 5 * 32)}
    if kind == "batch":
        fr = _uneven(c)
        return {"bytes": sum(4 * c["ne"] * (nt + 2 * nz) for nt, nz in fr),
                "flops": sum(_map_flops(c["ne"], nt, nz, len(_bins(c, nt)), c["ne"], 3) for nt, nz in fr)}
    ne, nt, nz, nb = c["ne"], c["nt"], c["nz"], len(_bins(c))
    nx = ne * (2 if c.get("pad2x") or c.get("upsample2x") else 1)
    out = nz * (2 * ne if c.get("upsample2x") else ne)
    apertures = {"as": 1, "dax": 2, "learned": 1}.get(kind, 3)
    maps = 1 if kind == "as" else 2 + (1 + (3 if apertures == 3 else 1) if c.get("all_maps") else 0)
    flops = _map_flops(ne, nt, nz, nb, nx, apertures)
    if kind == "learned":
        flops += nz * ne * 2.0 * 9 * (5 * 32 + 3 * 32 * 32 + 32)
    return {"bytes": n * 4 * (ne * nt + maps * out), "flops": n * flops}


# ------------------------------------------------------------- exact values --
def _phasors(c, bins, nt, nz, nx, pitch):
    """exp(i kz z) [bins][nz][nx]; evanescent components decay, or vanish where the case drops them."""
    dev = "cuda"
    k = torch.as_tensor(np.asarray(bins), device=dev, dtype=torch.float64) * (2 * np.pi * c["fs"] / nt / C)
    u = torch.arange(nx, device=dev, dtype=torch.float64)
    kx = torch.where(2 * u >= nx, u - nx, u) * (2 * np.pi / (nx * pitch))
    d = k[:, None] ** 2 - kx[None] ** 2
    kz = torch.sqrt(d.abs())[:, None, :] * (c["z0"] + torch.arange(nz, device=dev, dtype=torch.float64) * c["dz"])[None, :, None]
    live = d[:, None, :] >= 0
    amp = torch.where(live, torch.ones_like(kz), torch.exp(-kz) * (0.0 if c.get("evanescent_zero") else 1.0))
    return torch.polar(amp, torch.where(live, kz, torch.zeros_like(kz)))


def _aperture_sums(c, rf, bins, nz, apod, cache, bands=1):
    """Sums over the bins of |p_q|^2 and Re conj(p_q) p_r, per band of bins: [bands][6 or 3 or 1][nz][nx]."""
    ne, nt = rf.shape
    wide = 2 if c.get("pad2x") or c.get("upsample2x") else 1
    nx, pitch = ne * wide, PITCH / (2 if c.get("upsample2x") else 1)
    S = torch.fft.rfft(rf.double(), dim=1)[:, torch.as_tensor(np.asarray(bins), device="cuda")].T      # [bins][ne]
    src = torch.zeros((len(bins), len(apod), nx), device="cuda", dtype=torch.complex128)
    at = slice(0, 2 * ne, 2) if c.get("upsample2x") else slice(0, ne)
    src[:, :, at] = S[:, None, :] * apod[None]
    V = torch.fft.fft(src, dim=2)
    pairs = {1: [], 2: [(0, 1)], 3: [(0, 1), (1, 2), (2, 0)]}[len(apod)]
    out = torch.zeros((bands, len(apod) + len(pairs), nz, nx), device="cuda", dtype=torch.float64)
    nb = len(bins)
    step = max(1, (1 << 24) // (nz * nx))
    edges = [nb * b // bands for b in range(bands + 1)]
    for b in range(bands):
        for k0 in range(edges[b], edges[b + 1], step):
            k1 = min(edges[b + 1], k0 + step)
            if (k0, k1) not in cache:
                cache[k0, k1] = _phasors(c, bins[k0:k1], nt, nz, nx, pitch)
            p = [torch.fft.ifft(V[k0:k1, q, None, :] * cache[k0, k1], dim=2) for q in range(len(apod))]
            for i, f in enumerate(p):
                out[b, i] += (f.real ** 2 + f.imag ** 2).sum(0)
            for i, (q, r) in enumerate(pairs):
                out[b, len(apod) + i] += (p[q].real * p[r].real + p[q].imag * p[r].imag).sum(0)
    return out


def _weights(sums, n):
    """Clamped pair NCCs, rho before the max normalisation, and the coherent energy."""
    a, x = sums[:n], sums[n:]
    pairs = [(0, 1), (1, 2), (2, 0)][:3 if n == 3 else 1]
    rho = []
    for v, (q, r) in zip(x, pairs):
        den = torch.sqrt(a[q]) * torch.sqrt(a[r])
        rho.append(torch.where(den > 0, v / den, torch.full_like(v, EPS)).clamp_min(EPS))
    rho = torch.stack(rho)
    return rho, rho[0] if n == 2 else rho.prod(0) ** (1 / 3), (a.sum(0) + 2 * x.sum(0)).clamp_min(0)


def _pattern(c, n):
    return torch.stack([((torch.arange(c["ne"], device="cuda") // c["pattern"]) % n == q).double() for q in range(n)])


def _layers():
    p, o, out = torch.from_numpy(learn.load_checkpoint()[0]).cuda().double(), 0, []
    for ci, co in ((5, 32), (32, 32), (32, 32), (32, 32), (32, 1)):
        n = 9 * ci * co
        out += [p[o:o + n].view(co, ci, 3, 3).clone().requires_grad_(), p[o + n:o + n + co].clone().requires_grad_()]
        o += n + co
    return out


def _network(x, layers):
    for k in range(5):
        # the 3x3 correlation as nine matrix products (64-bit convolutions are slow in the libraries)
        n, ci, h, w = x.shape
        pad = torch.nn.functional.pad(x, (1, 1, 1, 1))
        x = sum(torch.einsum("oc,nchw->nohw", layers[2 * k][:, :, u, v], pad[:, :, u:u + h, v:v + w])
                for u in range(3) for v in range(3)) + layers[2 * k + 1].view(1, -1, 1, 1)
        x = torch.relu(x) if k < 4 else x
    return EPS + (1 - EPS) * torch.sigmoid(x[:, 0])


def _exact_grads(c, seed):
    feats, target = _training_batch(c, seed)
    nz, nx, n = c["nz"], c["ne"], c["frames"]
    layers = _layers()
    loss = torch.zeros((), device="cuda", dtype=torch.float64)
    for f in range(n):
        x = feats[f].view(torch.bfloat16).view(1, nz + 2, nx + 2, 8)[:, 1:-1, 1:-1, :5].permute(0, 3, 1, 2).double()
        w = WEIGHT_FLOOR + (1 - WEIGHT_FLOOR) * (10 ** (4 * x[:, 0]) - FEATURE_FLOOR).clamp(0, 1)
        part = (w * (_network(x, layers) - target[f:f + 1].double()) ** 2).sum() / (n * nz * nx)
        part.backward()
        loss += part.detach()
    return {"grads": torch.cat([p.grad.reshape(-1) for p in layers]), "loss": loss.view(1)}


def _exact_learned(c, rf):
    """Network on the band energies, the gate on the 32-row tile of the predicted peak, the method where it fails."""
    bins, nz, ne = _bins(c), c["nz"], c["ne"]
    ones, apod, cache, res = torch.ones((1, ne), device="cuda", dtype=torch.float64), _pattern(c, 3), {}, []
    layers = [p.detach() for p in _layers()]
    banded, plain = {}, {}
    for f in range(c["frames"]):
        bands = _aperture_sums(c, rf[f], bins, nz, ones, banded, bands=4)[:, 0]
        e = bands.sum(0)
        x = torch.log10(torch.cat([e[None], bands]) / e.max() + FEATURE_FLOOR) / 4
        rho = _network(x[None], layers)[0]
        _, rx, ex = _weights(_aperture_sums(c, rf[f], bins, nz, apod, plain)[0], 3)
        row = int((rho ** 2 * e).argmax()) // ne // 32 * 32
        ip, ix = (rho ** 2 * e)[row:row + 32], (rx ** 2 * ex)[row:row + 32]
        err = torch.linalg.norm(ip - ix) / torch.linalg.norm(ix)
        r, g = (rho, e) if float(err) <= c["gate"] else (rx, ex)
        rn = r / r.max()
        res.append((rn ** 2 * g, rn, err))
    return {"image": torch.stack([r[0] for r in res]), "rho_n": torch.stack([r[1] for r in res]),
            "gate_err": torch.stack([r[2] for r in res]), "gate_pass": None}


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "grads":
        return _exact_grads(c, seed)
    rf = _frames(c, seed)
    if kind == "learned":
        return _exact_learned(c, rf)
    if kind == "batch":
        img, rho = [], []
        for f, (nt, nz) in enumerate(_uneven(c)):
            _, r, e = _weights(_aperture_sums(c, rf[f], _bins(c, nt), nz, _pattern(c, 3), {})[0], 3)
            r = r / r.max()
            for to, v in ((img, r * r * e), (rho, r)):
                to.append(v.reshape(-1))
        return {"image": torch.cat(img), "rho_n": torch.cat(rho)}
    bins, cache, outs = _bins(c), {}, []
    crop = c["ne"] if c.get("pad2x") else None
    for f in range(c["frames"]):
        n = {"as": 1, "dax": 2}.get(kind, 3)
        apod = torch.ones((1, c["ne"]), device="cuda", dtype=torch.float64) if n == 1 else _pattern(c, n)
        sums = _aperture_sums(c, rf[f], bins, c["nz"], apod, cache)[0][:, :, :crop]
        if n == 1:
            outs.append({"energy": sums[0]})
            continue
        pairs, r, e = _weights(sums, n)
        r = r / r.max()
        o = {"image": r * r * e, "rho_n": r}
        if c.get("all_maps"):
            o.update(rho_pairs=pairs, image_as=e)
        outs.append(o)
    out = {k: torch.stack([o[k] for o in outs]) for k in outs[0]}
    return {k: v.cpu().numpy() for k, v in out.items()} if kind == "host" else out
