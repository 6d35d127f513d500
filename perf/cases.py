"""The work that users of this framework have it do, as cases that a timing program can run.

A case is one call (or one short sequence of calls) of the public Python API
(``paper_2206_09151_gb300.recon``) at one problem size: whole reconstructions
(``Reconstructor.run``), the two stages on their own (``filter_stage``, ``backproject``), a batch of
uneven tomograms (``Batch.run``), the two 3D-Fourier forms (``swap_ct`` + ``swap_phase``,
``grid_run``) and the training of the learned regulariser (``train_mlp``).  Whole runs keep the
default float32 layer stacks; the bfloat16 stacks of the large scans are measured at the two
stages that write and read them.

``exact`` computes the same outputs in 64 bits with plain torch, from the formulas that
``include/recon.h`` states."""
from __future__ import annotations

import math
import os
import random

import numpy as np
import torch

import paper_2206_09151_gb300 as package
from paper_2206_09151_gb300.recon import Batch, Reconstructor, train_mlp

# Wavelength, pitch (m), beta/delta, Tikhonov eps, Cs (m), counts per pixel, defocus range (m).
PHYSICS = {
    "xray": dict(lam=1e-10, delta=1e-9, sigma=0.01, eps=1e-2, cs=0.0, photons=1e4, defocus=(100e-9, 120e-9)),
    "electron": dict(lam=1.97e-12, delta=1e-10, sigma=0.07, eps=0.1, cs=2.7e-3, photons=100.0, defocus=(0.5e-6, 1.5e-6)),
    "electron_fine": dict(lam=1.97e-12, delta=5e-11, sigma=0.07, eps=0.1, cs=2.7e-3, photons=50.0,
                          defocus=(0.75e-6, 1.25e-6)),
}
INTENSITY_FLOOR = 1e-6  # images are I / I_in, floored before the logarithm
FIXED = float(1 << 24)  # depth coordinates are rounded to 2^-24 layer
HIDDEN = 64             # width of the regulariser network
PARAMS = 3 * HIDDEN + HIDDEN + HIDDEN * HIDDEN + HIDDEN + HIDDEN + 1


def _case(name, kind, **kw):
    case = dict(kind=kind, geometry="axis", nx=64, ny=64, nz=64, nu=64, nv=64, views=90, span_deg=180.0, layers=8,
                filter="tikhonov", stack="f32", interp="nearest", input="intensity", physics="xray", count=0,
                tomograms=0, mix=0, steps=0, noise_filter=False)
    case.update(kw)
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # a quick look during alignment, or one of many small soft X-ray scans: launches and latency
        _case("small_scan", "run"),
        # an ordinary atomic-resolution electron tomogram
        _case("mid_scan", "run", nx=256, ny=256, nz=256, nu=256, nv=256, views=360, layers=32, physics="electron"),
        # odd sizes throughout, views over the full turn with the opposite-pair filter; the volume's
        # rows fall between two detector rows
        _case("ragged_pair_scan", "run", nx=151, ny=133, nz=141, nu=157, nv=144, views=151, span_deg=360.0, layers=11,
              filter="pair"),
        # conventional filtered backprojection of ready contrasts: one layer, no phase retrieval
        _case("fbp_scan", "run", nx=512, ny=256, nz=512, nu=512, nv=256, views=360, layers=1, filter="off",
              input="contrast"),
        # an arbitrary geometry (random views in a cone, sampling-density weights) with the layer blend
        _case("cone_blend_scan", "run", geometry="cone", nx=160, ny=160, nz=96, nu=192, nv=192, views=200, layers=16,
              interp="linear", physics="electron"),
        # the largest images: one sub-scan's layer stacks of the 1024 x 1024 x 256 slab, bfloat16
        _case("slab_filter", "filter", geometry="cone", nx=1024, ny=1024, nz=256, nu=1024, nv=1024, views=240, layers=64,
              stack="bf16", physics="electron_fine", count=12),
        # ... and their backprojection into the slab
        _case("slab_backproject", "backproject", geometry="cone", nx=1024, ny=1024, nz=256, nu=1024, nv=1024, views=240,
              layers=64, stack="bf16", physics="electron_fine", count=24),
        # layer stacks of the 512^3 scan with the trained regulariser choosing eps
        _case("learned_filter", "filter", nx=512, ny=512, nz=512, nu=512, nv=512, views=720, layers=64, filter="mlp",
              stack="bf16", physics="electron", count=30),
        # a service that reconstructs uneven tomograms together
        _case("uneven_batch", "batch", tomograms=8, mix=4001),
        # Eq. 12: the CT step once, then the phase step for two values of beta/delta
        _case("swapped_order", "swap", nx=256, ny=256, nz=256, nu=256, nv=256, views=120, span_deg=360.0, layers=32,
              filter="pair", physics="electron"),
        # the Fourier-gridding reconstruction with its noise filter
        _case("fourier_gridding", "grid", nx=192, ny=192, nz=192, nu=192, nv=192, views=180, physics="electron",
              noise_filter=True),
        # a mini-batch of the regulariser's training (forward, backward, Adam)
        _case("regulariser_training", "train", nx=128, ny=128, nz=128, nu=128, nv=128, views=32, layers=16,
              physics="electron", steps=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges that the listed ones stand for (cost at most the largest listed one's)."""
    kind = rng.choice(["run", "run", "run", "run", "filter", "filter", "backproject", "backproject", "batch", "swap",
                       "grid", "train"])
    physics = rng.choice(["xray", "electron"])
    if kind == "batch":
        return _case(None, kind, tomograms=rng.randint(3, 8), mix=rng.randint(1, 10 ** 6))
    if kind == "train":
        n = _log_int(rng, 24, 128)
        return _case(None, kind, nx=n, ny=n, nz=n, nu=n, nv=n, views=rng.randint(8, 32), layers=rng.randint(4, 16),
                     physics=physics, steps=rng.randint(1, 6))
    if kind in ("swap", "grid"):
        n = _log_int(rng, 40, 224)
        case = _case(None, kind, nx=n, ny=int(n * rng.uniform(0.7, 1.0)), nz=int(n * rng.uniform(0.5, 1.0)),
                     nu=n, nv=int(n * rng.uniform(0.8, 1.0)), views=_log_int(rng, 24, 180), layers=_log_int(rng, 2, 32),
                     span_deg=360.0 if kind == "swap" else 180.0, physics=physics,
                     filter="pair" if kind == "swap" else "tikhonov",
                     noise_filter=kind == "grid" and rng.random() < 0.5)
    else:
        geometry = rng.choice(["axis", "axis", "cone", "cone", "tilted"])
        filt = rng.choice(["tikhonov", "tikhonov", "pair", "off", "mlp"])
        n = _log_int(rng, 32, 320 if kind == "run" else 1024)
        deep = rng.uniform(0.25, 1.0) if kind != "run" else rng.uniform(0.5, 1.0)
        case = _case(None, kind, geometry=geometry, nx=n, ny=int(n * rng.uniform(0.6, 1.0)), nz=max(8, int(n * deep)),
                     nu=min(1024, max(17, int(n * rng.uniform(0.9, 1.2)))),
                     nv=min(1024, max(17, int(n * rng.uniform(0.6, 1.2)))), views=_log_int(rng, 24, 360),
                     span_deg=360.0 if filt == "pair" else 180.0, layers=1 if filt == "off" else _log_int(rng, 2, 64),
                     filter=filt, interp=rng.choice(["nearest", "nearest", "linear"]),
                     input=rng.choice(["intensity", "intensity", "contrast"]),
                     stack="f32" if kind == "run" else rng.choice(["bf16", "bf16", "f32"]), physics=physics)
        if kind != "run":
            case["count"] = min(case["views"], rng.randint(4, 24))
    cap = max(work(c)["flops"] for c in listed() if c["kind"] == kind)
    while work(case)["flops"] > cap:
        case["views"] = max(1, int(0.8 * case["views"]))
        if case["count"]:
            case["count"] = max(1, min(case["views"], int(0.8 * case["count"])))
        case["layers"] = max(1, int(0.9 * case["layers"]))
    return case


# ----------------------------------------------------------------------------- inputs
def _members(case):
    """The tomograms of a batch: grids n^3 with n in {64, 96, ..., 256}, 60 to 180 views, 4 to 32 layers."""
    rng = random.Random(case["mix"])
    out = []
    for _ in range(case["tomograms"]):
        n = rng.choice(range(64, 257, 32))
        out.append(_case(None, "run", nx=n, ny=n, nz=n, nu=n, nv=n, views=rng.randint(60, 180), layers=rng.randint(4, 32),
                         physics=rng.choice(["xray", "electron"])))
    return out


def _padded(n):
    p = 1
    while p < 2 * n:
        p *= 2
    return p


def _axis_rotations(views, span, start):
    th = start + span * np.arange(views) / views
    rot = np.zeros((views, 3, 3))
    rot[:, 0, 0], rot[:, 0, 2] = np.cos(th), np.sin(th)
    rot[:, 1, 1] = 1.0
    rot[:, 2, 0], rot[:, 2, 2] = -np.sin(th), np.cos(th)
    return rot


def _rotations(case, rng):
    """(views, 3, 3): about the volume's y axis, about an axis tilted out of it, or random in a 60-degree cone."""
    if case["geometry"] == "cone":
        out = []
        while len(out) < case["views"]:
            q, r = np.linalg.qr(rng.standard_normal((256, 3, 3)))
            q = q * np.sign(np.einsum("nii->ni", r))[:, None, :]
            q[:, 0] *= np.sign(np.linalg.det(q))[:, None]
            out += list(q[np.abs(q[:, 2, 2]) >= 0.5])
        return np.stack(out[:case["views"]])
    rot = _axis_rotations(case["views"], math.radians(case["span_deg"]), rng.uniform(0.0, 1.0))
    if case["geometry"] == "tilted":
        c, s = math.cos(0.35), math.sin(0.35)
        rot = rot @ np.array([[1.0, 0.0, 0.0], [0.0, c, -s], [0.0, s, c]])
    return rot


def _scan(case, seed):
    """Rotations, defocus of each view and images of one scan: seeded Gaussian blobs in the volume,
    their projections as contrasts, Poisson counts at the dose."""
    p = PHYSICS[case["physics"]]
    rng = np.random.default_rng(seed)
    rot = _rotations(case, rng)
    D, nu, nv = case["views"], case["nu"], case["nv"]
    defocus = rng.uniform(*p["defocus"], D)
    if case["kind"] == "swap":  # Eq. 12 holds for one defocus
        defocus[:] = defocus[0]
    K = 48
    size = np.array([case["nx"], case["ny"], case["nz"]], float)
    centre = torch.tensor(rng.uniform(-0.35, 0.35, (K, 3)) * size, dtype=torch.float32, device="cuda")
    weight = torch.tensor(rng.uniform(0.01, 0.06, K), dtype=torch.float32, device="cuda")
    width = torch.tensor(rng.uniform(1.0, 0.04 * max(nu, nv) + 1.0, K), dtype=torch.float32, device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(seed)
    images = torch.empty((D, nv, nu), dtype=torch.float32, device="cuda")
    R = torch.tensor(rot, dtype=torch.float32, device="cuda")
    u = torch.arange(nu, device="cuda") - (nu - 1) / 2
    v = torch.arange(nv, device="cuda") - (nv - 1) / 2
    for a in range(0, D, 32):
        b = min(D, a + 32)
        pu, pv = (R[a:b, 0] @ centre.T)[:, :, None], (R[a:b, 1] @ centre.T)[:, :, None]
        gu = torch.exp(-0.5 * ((u - pu) / width[:, None]) ** 2)
        gv = torch.exp(-0.5 * ((v - pv) / width[:, None]) ** 2) * weight[:, None]
        contrast = -torch.bmm(gv.transpose(1, 2), gu)
        counts = torch.poisson(torch.exp(contrast) * p["photons"], generator=gen)
        image = counts / p["photons"]
        images[a:b] = torch.log(image.clamp_min(0.5 / p["photons"])) if case["input"] == "contrast" else image
    return rot, defocus, images


def _weights():
    """The trained regulariser that the package ships."""
    with np.load(os.path.join(os.path.dirname(package.__file__), "data", "regulariser.npz")) as f:
        return f["weights"].astype(np.float32)


def _reconstructor(case, rot, defocus, **kw):
    p = PHYSICS[case["physics"]]
    if case["filter"] == "mlp":
        kw.update(mlp_weights=_weights(), nsr=p["photons"] ** -0.5, mlp_views=case["views"])
    return Reconstructor(rot, case["nu"], case["nv"], (case["nx"], case["ny"], case["nz"]), lam=p["lam"],
                         delta=p["delta"], defocus=defocus, nz_layers=case["layers"], sigma=p["sigma"], eps=p["eps"],
                         cs=p["cs"], filter=case["filter"], input_mode=case["input"], stack_dtype=case["stack"],
                         ramp="density" if case["geometry"] == "cone" else "single_axis", layer_interp=case["interp"],
                         **kw)


def _layers_of(case, seed, su):
    """A block of layer stacks Y (count, layers, nv, nu): noise, as the filtered images of a low-dose scan
    are, in the stack's type and the tap-pair layout (rows ``su`` entries apart)."""
    dt = torch.bfloat16 if case["stack"] == "bf16" else torch.float32
    nu, nv, L = case["nu"], case["nv"], case["layers"]
    gen = torch.Generator(device="cuda").manual_seed(seed + 77)
    pairs = torch.zeros((case["count"], L, nv + 2, su, 2), dtype=dt, device="cuda")
    for n in range(case["count"]):
        y = torch.randn((L, nv, nu), generator=gen, device="cuda").to(dt)
        pairs[n, :, 1:nv + 1, 1:nu + 1, 0] = y
        pairs[n, :, 1:nv + 1, :nu, 1] = y
    return pairs


def _targets(case, seed):
    """Layer projections (metres) that a training image is fitted to: smooth seeded fields."""
    gen = torch.Generator(device="cuda").manual_seed(seed + 99)
    p = PHYSICS[case["physics"]]
    coarse = torch.rand((case["views"], case["layers"], 12, 12), generator=gen, device="cuda")
    fine = torch.nn.functional.interpolate(coarse, size=(case["nv"], case["nu"]), mode="bilinear", align_corners=False)
    return (fine * (0.02 * p["lam"] / case["layers"])).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        scans = [(m, *_scan(m, seed + 1000 * q)) for q, m in enumerate(_members(case))]
        recons = [_reconstructor(m, rot, defocus, allocate=False) for m, rot, defocus, _ in scans]
        return dict(kind=kind, batch=Batch(recons), images=[s[3] for s in scans], volumes=[r.new_volume() for r in recons])
    rot, defocus, images = _scan(case, seed)
    if kind == "train":
        p = PHYSICS[case["physics"]]
        kw = dict(nz_layers=case["layers"], lam=p["lam"], delta=p["delta"], sigma=p["sigma"], cs=p["cs"],
                  nsr=p["photons"] ** -0.5, steps=case["steps"], lr=3e-3, adam_step=0)
        return dict(kind=kind, weights=_weights(), images=images, targets=_targets(case, seed), rot=rot, defocus=defocus,
                    grid=(case["nx"], case["ny"], case["nz"]), kw=kw)
    r = _reconstructor(case, rot, defocus, dir_block=case["count"], allocate=kind not in ("swap", "grid"))
    state = dict(kind=kind, recon=r, images=images, volume=r.new_volume() if kind != "filter" else None,
                 count=case["count"], physics=PHYSICS[case["physics"]], noise_filter=case["noise_filter"])
    if kind == "backproject":
        state["stack"] = _layers_of(case, seed, r.stack_row_stride)[:, :, :, :case["nu"] + 1, :]
    return state


def run(state):
    kind = state["kind"]
    if kind == "batch":
        return state["batch"].run(state["images"], state["volumes"])
    if kind == "train":
        adam = np.zeros(2 * PARAMS, np.float32)
        weights, loss, _ = train_mlp(state["weights"], state["images"], state["targets"], state["rot"], state["defocus"],
                                     state["grid"], adam_state=adam, **state["kw"])
        return dict(weights=weights, loss=loss, adam=adam)
    r, p = state["recon"], state["physics"]
    if kind == "run":
        return r.run(state["images"], state["volume"])
    if kind == "filter":
        return r.filter_stage(state["images"], 0, state["count"])
    if kind == "backproject":
        return r.backproject(state["stack"], 0, state["count"], state["volume"], False)
    if kind == "swap":
        spectrum = r.swap_ct(state["images"])
        return [r.swap_phase(spectrum, p["sigma"], p["eps"], state["volume"]), r.swap_phase(spectrum, 0.0, p["eps"])]
    return r.grid_run(state["images"], p["photons"] ** -0.5 if state["noise_filter"] else 0.0, state["volume"])


# ----------------------------------------------------------------------------- work
def work(case):
    """Bytes in and out once each; flops of the real 2D transforms (5/2 N log2 N each), 4 per filtered
    coefficient and 11 per sampled voxel (coordinates, two row lerps, one column lerp, the sum)."""
    kind = case["kind"]
    if kind == "batch":
        parts = [work(m) for m in _members(case)]
        return {k: sum(q[k] for q in parts) for k in ("bytes", "flops")}
    P, L = _padded(max(case["nu"], case["nv"])), case["layers"]
    views = case["count"] or case["views"]
    nvox, image = case["nx"] * case["ny"] * case["nz"], 4 * case["nu"] * case["nv"]
    fft2 = 2.5 * P * P * math.log2(P * P)
    stack = L * (case["nv"] + 2) * (case["nu"] + 1) * (4 if case["stack"] == "bf16" else 8)
    stage_a = fft2 + L * (fft2 + 2.0 * P * P)
    stage_b = (22.0 if case["interp"] == "linear" else 11.0) * nvox
    if kind == "filter":
        return {"bytes": views * (image + stack), "flops": views * stage_a}
    if kind == "backproject":
        return {"bytes": views * stack + 4 * nvox, "flops": views * stage_b}
    if kind == "train":
        return {"bytes": views * image * (1 + L), "flops": views * (1 + L) * fft2 + case["steps"] * views * L * 20.0 * P * P}
    cells = _padded(case["nx"]) * _padded(case["ny"]) * _padded(case["nz"])
    fft3 = 2.5 * cells * math.log2(cells)
    if kind == "swap":
        return {"bytes": views * image + 2 * 4 * nvox, "flops": 2 * views * (stage_a + stage_b) + 4 * fft3 + 40.0 * cells}
    if kind == "grid":
        return {"bytes": views * image + 4 * nvox, "flops": views * (fft2 + 60.0 * P * P) + fft3 + 10.0 * cells}
    return {"bytes": views * image + 4 * nvox, "flops": views * (stage_a + stage_b)}


# ----------------------------------------------------------------------------- 64 bits
F64 = dict(dtype=torch.float64, device="cuda")


def _signed(P):
    m = torch.arange(P, **F64)
    return torch.where(m < P // 2, m, m - P)


def _half_grid(P):
    """Signed frequencies (m_v, m_u) of the half spectrum that rfft2 gives."""
    mu = torch.arange(P // 2 + 1, **F64)
    return _signed(P)[:, None].expand(P, P // 2 + 1), mu[None, :].expand(P, P // 2 + 1)


def _spectrum(case, image, P):
    g = image.double()
    if case["input"] == "intensity":
        g = torch.log(torch.clamp_min(g, INTENSITY_FLOOR))
    return torch.fft.rfft2(g, s=(P, P))


def _ramp(P, delta, views):
    n = _signed(P)
    h = torch.where(n.remainder(2) == 1, -1.0 / (n.abs().clamp_min(1.0) ** 2 * math.pi ** 2 * delta ** 2),
                    torch.zeros_like(n))
    h[0] = 1.0 / (4.0 * delta * delta)
    return math.pi / views * delta * torch.fft.fft(h).real[:P // 2 + 1]


def _corners(q):
    """The 8 cells around each point of q (N, 3) and their trilinear weights."""
    base = torch.floor(q)
    f = q - base
    base = base.long()
    for dz in (0, 1):
        for dy in (0, 1):
            for dx in (0, 1):
                w = (f[:, 0] if dx else 1 - f[:, 0]) * (f[:, 1] if dy else 1 - f[:, 1]) * (f[:, 2] if dz else 1 - f[:, 2])
                yield base[:, 0] + dx, base[:, 1] + dy, base[:, 2] + dz, w


class _Density:
    """Sampling density of every view's DFT samples, and the weight that divides by it."""

    def __init__(self, rot, P, delta):
        s = max(1, P // 128)
        Gh = int(math.ceil(math.sqrt(2.0) * (P / 2) / s)) + 2
        G = 2 * Gh + 1
        self.rot, self.P, self.s, self.Gh, self.G = torch.tensor(rot, **F64), P, s, Gh, G
        S = torch.zeros(G ** 3, **F64)
        m = torch.arange(-P // 2, P // 2, s, **F64)
        mu, mv = (x.reshape(-1, 1) for x in torch.meshgrid(m, m, indexing="ij"))
        for R in self.rot:
            q = (mu * R[0] + mv * R[1]) / s
            for sign in (1.0, -1.0):
                for x, y, z, w in _corners(sign * q):
                    S.index_add_(0, ((z + Gh) * G + y + Gh) * G + x + Gh, w * (0.5 * s * s))
        c = (torch.arange(G, device="cuda") - Gh) ** 2
        band = (c[:, None, None] + c[None, :, None] + c[None, None, :]) <= (Gh - 2) ** 2
        self.S, self.eps = S, 1e-3 * S[band.reshape(-1)].sum() / band.sum()
        self.g = s ** 3 / (P * delta)

    def at(self, n, mv, mu):
        q = (mu.reshape(-1, 1) * self.rot[n, 0] + mv.reshape(-1, 1) * self.rot[n, 1]) / self.s
        val = torch.zeros(q.shape[0], **F64)
        for x, y, z, w in _corners(q):
            val += w * self.S[((z + self.Gh) * self.G + y + self.Gh) * self.G + x + self.Gh]
        return (self.g / (val + self.eps)).reshape(mu.shape)

    def weight(self, n):
        """On the Nyquist bins, which stand for two frequencies, the mean over both."""
        P = self.P
        mv, mu = _half_grid(P)
        edge_u, edge_v = mu == P // 2, mv == -(P // 2)
        w0 = self.at(n, mv, mu)
        w1 = self.at(n, torch.where(edge_v & ~edge_u, -mv, mv), torch.where(edge_u, -mu, mu))
        return torch.where(edge_u | edge_v, 0.5 * (w0 + w1), w0)


def _bins(P):
    """Radial bin of each half-spectrum frequency, and the number of bins."""
    width = max(1, P // 128)
    nb = math.isqrt(P * P // 2) // width + 1
    mv, mu = _half_grid(P)
    sq = (mv * mv + mu * mu).long()
    r = torch.sqrt(sq.double()).long()
    r = torch.where(r * r > sq, r - 1, r)
    r = torch.where((r + 1) * (r + 1) <= sq, r + 1, r)
    return (r // width).clamp_max(nb - 1), nb, width


def _features(case, G, P, z, defocus):
    """Inputs of the regulariser network for each (layer, radial bin) of one image."""
    p = PHYSICS[case["physics"]]
    bins, nb, width = _bins(P)
    mult = torch.full_like(G.real, 2.0)
    mult[:, 0] = mult[:, -1] = 1.0
    power = torch.zeros(nb, **F64).index_add_(0, bins.reshape(-1), (mult * G.abs() ** 2).reshape(-1))
    count = torch.zeros(nb, **F64).index_add_(0, bins.reshape(-1), mult.reshape(-1))
    floor = case["nu"] * case["nv"] / p["photons"]
    snr = torch.clamp_min(power / count.clamp_min(1.0) - floor, 1e-3 * floor) / floor
    x = torch.empty((len(z), nb, 3), **F64)
    x[:, :, 0] = torch.clamp(torch.log10(snr), -3.0, 6.0) / 3.0
    x[:, :, 1] = (torch.arange(nb, **F64) + 0.5) * width / (P / 2)
    x[:, :, 2] = (p["lam"] * (defocus - z) / p["delta"] ** 2 / 100.0)[:, None]
    return x


def _network(theta, x):
    a, b, c, d, e = (HIDDEN * k for k in (3, 4, 4 + HIDDEN, 5 + HIDDEN, 6 + HIDDEN))
    h = torch.relu(x @ theta[:a].reshape(HIDDEN, 3).T + theta[a:b])
    h = torch.relu(h @ theta[b:c].reshape(HIDDEN, HIDDEN).T + theta[c:d])
    return torch.nn.functional.softplus(h @ theta[d:e] + theta[e])


def _chi(case, q2, r):
    p = PHYSICS[case["physics"]]
    return math.pi * p["lam"] * r * q2 + 0.5 * math.pi * p["cs"] * p["lam"] ** 3 * q2 * q2 - math.atan(p["sigma"])


def _depths(case, rot):
    """Layer centres (views, layers) in metres."""
    ext = np.abs(rot[:, 2]) @ np.array([case["nx"], case["ny"], case["nz"]], float) * PHYSICS[case["physics"]]["delta"]
    k = np.arange(case["layers"])
    return torch.tensor(-ext[:, None] / 2 + (k + 0.5) * (ext[:, None] / case["layers"]), **F64)


def _view_stack(case, image, n, defocus, z, W, mode=None):
    """Layers (layers, nv, nu) of one view; ``mode``: "cos" or "sin" of the depth phase alone."""
    p = PHYSICS[case["physics"]]
    P = _padded(max(case["nu"], case["nv"]))
    G = _spectrum(case, image, P)
    mv, mu = _half_grid(P)
    q2 = (mu * mu + mv * mv) / (P * p["delta"]) ** 2
    pref = p["lam"] / (4.0 * math.pi * math.sqrt(1.0 + p["sigma"] ** 2))
    if case["filter"] == "mlp" and mode is None:
        eps_bins = _network(torch.tensor(_weights(), **F64), _features(case, G, P, z, defocus)) / case["views"]
        bins = _bins(P)[0]
    if case["filter"] == "pair" and mode is None:
        chi = _chi(case, q2, defocus)
        s, c = torch.sin(chi), torch.cos(chi)
        s, c = s / (s * s + p["eps"]), c / (c * c + p["eps"])
    GW = G * W
    out = torch.empty((len(z), case["nv"], case["nu"]), **F64)
    for k in range(len(z)):
        depth = math.pi * p["lam"] * z[k] * q2
        if mode is not None:
            F = torch.cos(depth) if mode == "cos" else torch.sin(depth)
        elif case["filter"] == "off":
            F = 1.0
        elif case["filter"] == "pair":
            F = pref * (s * torch.cos(depth) - c * torch.sin(depth))
        else:
            sn = torch.sin(_chi(case, q2, defocus - z[k]))
            F = pref * sn / (sn * sn + (eps_bins[k][bins] if case["filter"] == "mlp" else p["eps"]))
        out[k] = torch.fft.irfft2(GW * F, s=(P, P))[:case["nv"], :case["nu"]]
    return out


def _stacks(case, rot, defocus, images, views, mode=None):
    p = PHYSICS[case["physics"]]
    P = _padded(max(case["nu"], case["nv"]))
    dens = _Density(rot, P, p["delta"]) if case["geometry"] == "cone" else None
    ramp = _ramp(P, p["delta"], case["views"])
    z = _depths(case, rot)
    for n in range(views):
        yield n, _view_stack(case, images[n], n, float(defocus[n]), z[n], ramp if dens is None else dens.weight(n), mode)


def _add_view(case, vol, R, layers):
    """Adds one view's ``layers`` (L, nv, nu) to the volume: bilinear, zero outside the detector."""
    nx, ny, nz, L = case["nx"], case["ny"], case["nz"], case["layers"]
    nu, nv = case["nu"], case["nv"]
    pad = torch.zeros((L, nv + 2, nu + 2), **F64)
    pad[:, 1:-1, 1:-1] = layers
    pad = pad.reshape(-1)
    ext = (abs(R[2, 0]) * nx + abs(R[2, 1]) * ny) + abs(R[2, 2]) * nz
    scale = L / ext
    step = [R[2, a] * scale for a in range(3)]
    t0 = 0.5 * L - ((step[0] * (0.5 * (nx - 1)) + step[1] * (0.5 * (ny - 1))) + step[2] * (0.5 * (nz - 1)))
    T = [int(np.rint(v * FIXED)) for v in (t0, *step)]  # the layer is decided in exact integers
    i = torch.arange(nx, device="cuda")[None, None, :]
    j = torch.arange(ny, device="cuda")[None, :, None]
    chunk = max(1, (1 << 24) // (nx * ny))
    for k0 in range(0, nz, chunk):
        k = torch.arange(k0, min(nz, k0 + chunk), device="cuda")[:, None, None]
        x, y, z = i.double() - (nx - 1) / 2, j.double() - (ny - 1) / 2, k.double() - (nz - 1) / 2
        a = (x * float(R[0, 0]) + y * float(R[0, 1]) + z * float(R[0, 2]) + (nu - 1) / 2).clamp(-1.0, nu)
        b = (x * float(R[1, 0]) + y * float(R[1, 1]) + z * float(R[1, 2]) + (nv - 1) / 2).clamp(-1.0, nv)
        a0, b0 = torch.floor(a).clamp_max(nu - 1), torch.floor(b).clamp_max(nv - 1)
        fa, fb = a - a0, b - b0
        at = ((b0 + 1) * (nu + 2) + a0 + 1).long()
        t = T[0] + T[1] * i + T[2] * j + T[3] * k

        def sample(layer):
            q = at + layer * ((nv + 2) * (nu + 2))
            top = (1 - fa) * pad[q] + fa * pad[q + 1]
            bot = (1 - fa) * pad[q + nu + 2] + fa * pad[q + nu + 3]
            return (1 - fb) * top + fb * bot

        if case["interp"] == "nearest":
            vol[k0:k0 + chunk] += sample((t >> 24).clamp(0, L - 1))
        else:
            t = t - (1 << 23)
            low = t >> 24
            w = torch.where((low < 0) | (low >= L - 1), torch.zeros_like(a), (t - (low << 24)).double() / FIXED)
            low = low.clamp(0, L - 1)
            vol[k0:k0 + chunk] += (1 - w) * sample(low) + w * sample((low + 1).clamp_max(L - 1))


def _volume(case, rot, stacks):
    vol = torch.zeros((case["nz"], case["ny"], case["nx"]), **F64)
    for n, y in stacks:
        _add_view(case, vol, rot[n], y)
    return vol


def _sides(case):
    n = [case["nx"], case["ny"], case["nz"]]
    P3 = [_padded(q) for q in n]
    return n, P3, [(P3[a] - n[a]) // 2 for a in range(3)]


def _exact_swap(case, rot, defocus, images):
    p = PHYSICS[case["physics"]]
    n, P3, off = _sides(case)
    box = tuple(slice(off[a], off[a] + n[a]) for a in (2, 1, 0))
    spec = []
    for mode in ("cos", "sin"):
        full = torch.zeros((P3[2], P3[1], P3[0]), **F64)
        full[box] = _volume(case, rot, _stacks(case, rot, defocus, images, case["views"], mode))
        spec.append(torch.fft.rfftn(full))
        del full
    f = [_signed(P3[a]) / (P3[a] * p["delta"]) for a in range(3)]
    f[0] = torch.arange(P3[0] // 2 + 1, **F64) / (P3[0] * p["delta"])
    q2 = f[0][None, None, :] ** 2 + f[1][None, :, None] ** 2 + f[2][:, None, None] ** 2
    lam = p["lam"]
    qp2 = 2.0 * q2 / (torch.sqrt(1.0 + lam * lam * q2) + 1.0)
    out = []
    for sigma in (p["sigma"], 0.0):
        chi = math.pi * lam * float(defocus[0]) * qp2 + 0.5 * math.pi * p["cs"] * lam ** 3 * qp2 * qp2 - math.atan(sigma)
        s, c = torch.sin(chi), torch.cos(chi)
        F = s / (s * s + p["eps"]) * spec[0] - c / (c * c + p["eps"]) * spec[1]
        F *= lam / (4.0 * math.pi * math.sqrt(1.0 + sigma * sigma))
        out.append(torch.fft.irfftn(F, s=(P3[2], P3[1], P3[0]))[box].contiguous())
    return out


def _exact_grid(case, rot, defocus, images):
    p = PHYSICS[case["physics"]]
    n, P3, off = _sides(case)
    P = _padded(max(case["nu"], case["nv"]))
    lam, delta, cells = p["lam"], p["delta"], P3[0] * P3[1] * P3[2]
    acc = torch.zeros((cells, 2), **F64)
    raw = torch.zeros((cells, 2), **F64)
    S = torch.zeros(cells, **F64)
    m = _signed(P)
    mv, mu = (x.reshape(-1) for x in torch.meshgrid(m, m, indexing="ij"))
    q2 = (mu * mu + mv * mv) / (P * delta) ** 2
    about_centre = torch.polar(torch.ones_like(mu), math.pi / P * (mu * (case["nu"] - 1) + mv * (case["nv"] - 1)))
    pref = lam / (4.0 * math.pi * math.sqrt(1.0 + p["sigma"] ** 2))
    side = torch.tensor([P3[a] * delta for a in range(3)], **F64)
    for v in range(case["views"]):
        g = images[v].double()
        g = g if case["input"] == "contrast" else torch.log(torch.clamp_min(g, INTENSITY_FLOOR))
        G = torch.fft.fft2(g, s=(P, P)).reshape(-1) * about_centre
        chi = _chi(case, q2, float(defocus[v]))
        s, c = torch.sin(chi), torch.cos(chi)
        Z = pref * G * torch.complex(s / (s * s + p["eps"]), -c / (c * c + p["eps"]))
        R = torch.tensor(rot[v], **F64)
        q = (mu[:, None] * R[0] + mv[:, None] * R[1]) / (P * delta) - 0.5 * lam * q2[:, None] * R[2]
        for x, y, z, w in _corners(q * side):
            cell = ((z % P3[2]) * P3[1] + y % P3[1]) * P3[0] + x % P3[0]
            S.index_add_(0, cell, w)
            acc.index_add_(0, cell, torch.view_as_real(Z) * w[:, None])
            if case["noise_filter"]:
                raw.index_add_(0, cell, torch.view_as_real(G) * w[:, None])
    eps_s = 1e-3 * S[S > 0].mean()
    F = torch.view_as_complex(acc) / (S + eps_s)
    if case["noise_filter"]:
        level = p["photons"] ** -0.5 * math.sqrt(case["nu"] * case["nv"])
        keep = torch.view_as_complex(raw).abs() / (S + eps_s) >= level / torch.sqrt(S.clamp_min(1e-300))
        F = torch.where(keep & (S > 0), F, torch.zeros_like(F))
    F = F.reshape(P3[2], P3[1], P3[0]) / delta
    for a, shape in ((0, (1, 1, -1)), (1, (1, -1, 1)), (2, (-1, 1, 1))):
        turn = -2.0 * math.pi * _signed(P3[a]) * (off[a] + (n[a] - 1) / 2) / P3[a]
        F = F * torch.polar(torch.ones_like(turn), turn).reshape(shape)
    return torch.fft.ifftn(F).real[tuple(slice(off[a], off[a] + n[a]) for a in (2, 1, 0))].contiguous()


def _exact_training(case, rot, defocus, images, targets):
    p = PHYSICS[case["physics"]]
    P = _padded(max(case["nu"], case["nv"]))
    z = _depths(case, rot)
    bins = _bins(P)[0]
    mv, mu = _half_grid(P)
    q2 = (mu * mu + mv * mv) / (P * p["delta"]) ** 2
    mult = torch.full_like(q2, 2.0)
    mult[:, 0] = mult[:, -1] = 1.0
    pref = p["lam"] / (4.0 * math.pi * math.sqrt(1.0 + p["sigma"] ** 2))
    N = case["views"]
    G = [_spectrum(case, images[n], P) for n in range(N)]
    x = torch.stack([_features(case, G[n], P, z[n], float(defocus[n])) for n in range(N)])
    sin = [torch.stack([torch.sin(_chi(case, q2, float(defocus[n]) - zk)) for zk in z[n]]) for n in range(N)]
    T = [torch.fft.rfft2(targets[n].double(), s=(P, P)) for n in range(N)]
    den = sum(float((mult * t.abs() ** 2).sum()) for t in T)
    theta = torch.tensor(_weights(), **F64)
    m1, m2, history = torch.zeros_like(theta), torch.zeros_like(theta), []
    for step in range(1, case["steps"] + 1):
        theta.requires_grad_(True)
        eps = _network(theta, x)
        leaf = eps.detach().requires_grad_(True)
        loss = 0.0
        for n in range(N):  # image by image: the spectra of all layers at once are large
            H = pref * sin[n] / (sin[n] ** 2 + leaf[n][:, bins])
            part = (mult * (H * G[n] - T[n]).abs() ** 2).sum() / den
            part.backward()
            loss += float(part)
        (grad,) = torch.autograd.grad(eps, theta, leaf.grad)
        history.append(loss)
        theta = theta.detach()
        m1, m2 = 0.9 * m1 + 0.1 * grad, 0.999 * m2 + 0.001 * grad * grad
        theta = theta - 3e-3 * (m1 / (1 - 0.9 ** step)) / (torch.sqrt(m2 / (1 - 0.999 ** step)) + 1e-8)
    return dict(weights=theta.cpu().numpy(), loss=np.array(history), adam=torch.cat([m1, m2]).cpu().numpy())


def _exact_filter(case, rot, defocus, images):
    nu, nv = case["nu"], case["nv"]
    pairs = torch.zeros((case["count"], case["layers"], nv + 2, nu + 1, 2), **F64)
    for n, y in _stacks(case, rot, defocus, images, case["count"]):
        pairs[n, :, 1:-1, 1:, 0] = y
        pairs[n, :, 1:-1, :nu, 1] = y
    return pairs


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for q, m in enumerate(_members(case)):
            rot, defocus, images = _scan(m, seed + 1000 * q)
            out.append(_volume(m, rot, _stacks(m, rot, defocus, images, m["views"])))
        return out
    rot, defocus, images = _scan(case, seed)
    if kind == "run":
        return _volume(case, rot, _stacks(case, rot, defocus, images, case["views"]))
    if kind == "filter":
        return _exact_filter(case, rot, defocus, images)
    if kind == "backproject":
        su = (case["nu"] + 4) // 4 * 4
        pairs = _layers_of(case, seed, su)[:, :, 1:-1, 1:case["nu"] + 1, 0]
        return _volume(case, rot, ((n, pairs[n].double()) for n in range(case["count"])))
    if kind == "swap":
        return _exact_swap(case, rot, defocus, images)
    if kind == "grid":
        return _exact_grid(case, rot, defocus, images)
    return _exact_training(case, rot, defocus, images, _targets(case, seed))
