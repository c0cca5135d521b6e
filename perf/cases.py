"""Performance cases of the imaging library: the calls that a user's program makes, through the public Python
entry points, with inputs of the distributions they meet in use.

Kinds of cases (the field ``kind``):

* ``fb``      the plain PnP-FB imaging loop (``Plan.fb_run`` with the Haar denoiser) from a zero image;
* ``learned`` the same loop with the faceted residual CNN and the App. C rescaling;
* ``grad``    one data-fidelity gradient step (``Plan.grad_step``);
* ``dirty``   one forward and one adjoint application (model visibilities and a dirty image);
* ``cnn``     one application of the faceted CNN denoiser;
* ``sara``    one application of the uSARA denoiser (a fixed number of dual iterations);
* ``train``   one l1 training step of the CNN whose gradients the program reads;
* ``train_fne`` the same with the firm non-expansiveness penalty.

Visibilities are those of a 64-antenna track (a Gaussian core plus outer antennas out to 4 km, symmetric hour
angles) of point sources and Gaussian blobs with 40 dB of noise, summed directly per visibility, so they do not
depend on the library.  ``exact`` restates every path in double precision with torch and numpy only.
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch

import paper_2207_11336_gb300 as pnp
from paper_2207_11336_gb300.heuristics import alpha_for_denoiser
from paper_2207_11336_gb300.train_denoiser import load as load_weights

WEIGHTS = os.path.join(os.path.dirname(os.path.abspath(pnp.__file__)), "weights", "dncnn_C3_fne.npz")
CNN_FLOP_PER_PX = 2 * 9 * 64 + 6 * 2 * 9 * 64 * 64 + 2 * 9 * 64
DEV = "cuda"


def listed():
    return [
        # the small imaging problem (256^2, KB J = 7): a whole loop of launch-bound iterations
        dict(name="fb_256", kind="fb", n=256, K=512, M=200_000, supports="7", wspread=0.0, weights="c64",
             robust=False, blocks=1, stacks=1, holo=False, iters=50),
        # the wide-field problem: 4096^2 image, w folded into G, Briggs-weighted data in 64 blocks
        dict(name="fb_4096", kind="fb", n=4096, K=8192, M=6_000_000, supports="7,9,12,16", wspread=4.0,
             weights="c64", robust=True, blocks=64, stacks=1, holo=False, iters=4),
        # the gradient step alone, as a program with its own outer loop calls it: dense uv coverage
        dict(name="grad_2048", kind="grad", n=2048, K=4096, M=5_000_000, supports="7,9,12,16", wspread=4.0,
             weights="c64", robust=False, blocks=1, stacks=1, holo=False, iters=1),
        # the largest image, G in BF16 (one band of the two-band wide-field problem)
        dict(name="grad_8192_bf16", kind="grad", n=8192, K=16384, M=5_000_000, supports="7,8,8,9", wspread=2.0,
             weights="bf16", robust=True, blocks=1, stacks=1, holo=False, iters=1),
        # an image side that is no power of two: model visibilities, then a dirty image
        dict(name="dirty_1500", kind="dirty", n=1500, K=4096, M=1_000_003, supports="7,9,12,16", wspread=4.0,
             weights="c64", robust=True, blocks=1, stacks=1, holo=False, iters=1),
        # the w-stacking hybrid
        dict(name="fb_stacked_1024", kind="fb", n=1024, K=2048, M=2_000_000, supports="7,9,12,16", wspread=4.0,
             weights="c64", robust=True, blocks=1, stacks=4, holo=False, iters=10),
        # many rows per grid cell: the holographic form of the normal operator
        dict(name="fb_holo_256", kind="fb", n=256, K=512, M=2_000_000, supports="7", wspread=0.0, weights="c64",
             robust=False, blocks=1, stacks=1, holo=True, iters=50),
        # the learned loop on uneven facets
        dict(name="learned_1024", kind="learned", n=1024, K=2048, M=1_000_000, supports="7,9,12,16", wspread=4.0,
             weights="c64", robust=True, blocks=1, stacks=1, holo=False, iters=6, facets=4),
        # the faceted CNN denoiser on its own: 512^2 facets with a 32-pixel halo
        dict(name="cnn_2048", kind="cnn", n=2048, facets=4, even=True),
        # the uSARA denoiser on its own
        dict(name="sara_1024", kind="sara", n=1024, prox=10),
        # denoiser training: the l1 step, and the step with the penalty
        dict(name="train_16x256", kind="train", batch=16, size=256),
        dict(name="train_fne_8x128", kind="train_fne", batch=8, size=128, iters=4),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["fb", "fb", "fb", "grad", "dirty", "learned", "cnn", "cnn", "sara", "train", "train_fne"])
    if kind == "cnn":
        return dict(kind=kind, n=2 * int(_log(rng, 64, 1024)), facets=rng.choice([1, 2, 3, 4]), even=rng.random() < 0.4)
    if kind == "sara":
        return dict(kind=kind, n=16 * int(_log(rng, 8, 80)), prox=rng.choice([5, 10, 20]))
    if kind in ("train", "train_fne"):
        size = int(_log(rng, 40, 256))
        c = dict(kind=kind, batch=max(1, min(16, int(_log(rng, 1, 16)), 1_048_576 // (size * size))), size=size)
        if kind == "train_fne":
            c.update(batch=min(c["batch"], 8), iters=rng.choice([2, 4, 8]))
        return c
    n = 2 * int(_log(rng, 64, 1600 if kind != "learned" else 640))
    if rng.random() < 0.5:
        n = 1 << round(math.log2(n))
    K = 1 << max(7, math.ceil(math.log2(2 * n)))
    M = int(min(4_000_000, _log(rng, 0.2, 4.0) * n * n + 20_000))
    supports = rng.choice(["7", "7,9,12,16", "7,9,12,16", "7,8,8,9", "5"])
    wspread = 0.0 if "," not in supports else (4.0 if "16" in supports else 2.0)
    c = dict(kind=kind, n=n, K=K, M=M, supports=supports, wspread=wspread,
             weights="bf16" if supports == "7,8,8,9" and rng.random() < 0.6 else "c64",
             robust=rng.random() < 0.6, blocks=rng.choice([1, 1, 16]), stacks=1, holo=False, iters=1)
    if kind == "fb":
        c["iters"] = rng.choice([4, 10, 20])
        if wspread and rng.random() < 0.25:
            c.update(stacks=rng.choice([2, 3]), iters=4)
        elif K <= 1024 and not wspread and rng.random() < 0.5:
            c["holo"] = True
    if kind == "learned":
        c.update(iters=4, facets=rng.choice([1, 2, 4]), weights="c64")
    return c


# ------------------------------------------------------------------------------------------------ inputs
def _geometry(c, seed):
    """(omega, w, dl, J_per_row or None, data weights d or None, block, stack, centres) of the uv track."""
    rng = np.random.default_rng([seed, 11])
    n, K, M = c["n"], c["K"], c["M"]
    core = rng.normal(0.0, 300.0, (48, 2))
    r, th = 4000.0 * np.sqrt(rng.random(16)), 2.0 * np.pi * rng.random(16)
    enu = np.concatenate([core, np.stack([r * np.cos(th), r * np.sin(th)], 1)])
    lat, dec = np.deg2rad(-30.7), np.deg2rad(-60.0)
    X, Y, Z = -np.sin(lat) * enu[:, 1], enu[:, 0], np.cos(lat) * enu[:, 1]
    i, j = np.triu_indices(64, 1)
    bx, by, bz = X[j] - X[i], Y[j] - Y[i], Z[j] - Z[i]
    nt = -(-M // i.size)
    hours = 8.0 if not c["wspread"] else 12.0
    ha = np.deg2rad(15.0) * np.linspace(-hours / 2, hours / 2, nt)
    sh, ch = np.sin(ha)[:, None], np.cos(ha)[:, None]
    uv = np.empty((nt * i.size, 2))
    uv[:, 0] = (sh * bx + ch * by).ravel()
    uv[:, 1] = (-np.sin(dec) * ch * bx + np.sin(dec) * sh * by + np.cos(dec) * bz).ravel()
    uv = uv[:M]
    omega = uv * (0.8 * np.pi / np.sqrt((uv ** 2).sum(1).max()))
    w, dl, Jr, sup = np.zeros(M), 0.0, None, [int(s) for s in c["supports"].split(",")]
    stack, centres, d = None, None, None
    if c["wspread"]:
        w = ((np.cos(dec) * ch * bx - np.cos(dec) * sh * by + np.sin(dec) * bz).ravel()[:M]) / 0.214
        dl = float(np.sqrt(c["wspread"] / (np.abs(w).max() * n * K)))
        edges = np.quantile(np.abs(w[::7]), [0.25, 0.5, 0.75])
        res = np.abs(w)
        if c["stacks"] > 1:
            cuts = np.quantile(w[::7], np.linspace(0, 1, c["stacks"] + 1)[1:-1])
            stack = np.searchsorted(cuts, w, side="right").astype(np.int32)
            centres = np.array([0.5 * (w[stack == s].min() + w[stack == s].max()) for s in range(c["stacks"])])
            res = np.abs(w - centres[stack])
        Jr = np.asarray(sup, np.int8)[np.searchsorted(edges, res, side="right")]
    k = torch.from_numpy(np.rint(omega * (n / (2 * np.pi))).astype(np.int64)).to(DEV)
    cell, conj = (k % n)[:, 0] * n + (k % n)[:, 1], (-k % n)[:, 0] * n + (-k % n)[:, 1]
    if c["robust"]:  # Briggs weighting, robust parameter 0
        cnt = (torch.bincount(cell, minlength=n * n) + torch.bincount(conj, minlength=n * n)).double()[cell]
        d = torch.sqrt(1.0 / (1.0 + cnt * (25.0 / cnt.mean())))
    d2 = torch.ones(M, dtype=torch.float64, device=DEV) if d is None else d * d
    W = (torch.bincount(cell, d2, n * n) + torch.bincount(conj, d2, n * n)).view(1, 1, n, n)
    box = torch.nn.functional.avg_pool2d(torch.nn.functional.pad(W, (1, 1, 1, 1), "circular"), 3, 1) * 9
    L = 0.5 * n * n * float(box.max())  # a bound on ||Re Phi^H Phi|| from the densest uv cells
    block = None
    if c["blocks"] > 1:
        block = np.minimum((np.arctan2(omega[:, 1], omega[:, 0]) + np.pi) * (c["blocks"] / (2 * np.pi)),
                           c["blocks"] - 1).astype(np.int32)
    return dict(omega=omega, w=w, dl=dl, Jr=Jr, J=sup[0], d=None if d is None else d.cpu().numpy(), block=block,
                stack=stack, centres=centres, L=L)


def _sky(n, rng):
    P = min(200, 20 + n // 16)
    return (rng.integers(n // 8, n - n // 8, (P, 2)) - n // 2, 10.0 ** rng.uniform(-4, 0, P),
            rng.integers(n // 4, n - n // 4, (4, 2)) - n // 2, rng.uniform(1.5, 4.0, 4) * max(1.0, n / 512),
            10.0 ** rng.uniform(-3, -1, 4))


def _sky_image(n, sky):
    pos, flux, bpos, bs, bf = sky
    x = np.zeros((n, n), np.float32)
    np.add.at(x, (pos[:, 0] + n // 2, pos[:, 1] + n // 2), flux)
    t = torch.from_numpy(x).to(DEV)
    p = torch.arange(n, device=DEV, dtype=torch.float64) - n // 2
    for q, s, f in zip(bpos, bs, bf):
        t += (f * torch.outer(torch.exp(-(p - int(q[0])) ** 2 / (2 * s * s)),
                              torch.exp(-(p - int(q[1])) ** 2 / (2 * s * s)))).float()
    return t


def _data(c, g, seed):
    """(y complex64 on the device, tau of the weighted noise, sky): D (sum over the sources + noise)."""
    rng = np.random.default_rng([seed, 12])
    sky = _sky(c["n"], rng)
    pos, flux, bpos, bs, bf = sky
    om = torch.from_numpy(g["omega"]).to(DEV)
    rate = torch.from_numpy(np.pi * g["w"] * g["dl"] ** 2).to(DEV)
    y = torch.zeros(c["M"], dtype=torch.complex128, device=DEV)
    for q, f in zip(pos, flux):
        ph = rate * float(q @ q) - om[:, 0] * float(q[0]) - om[:, 1] * float(q[1])
        y += torch.polar(torch.full_like(ph, float(f)), ph)
    r2 = (om ** 2).sum(1)
    for q, s, f in zip(bpos, bs, bf):
        ph = rate * float(q @ q) - om[:, 0] * float(q[0]) - om[:, 1] * float(q[1])
        y += torch.polar(float(f * 2 * np.pi * s * s) * torch.exp(-0.5 * s * s * r2), ph)
    tau = float(y.abs().square().mean().sqrt()) / 100.0
    gen = torch.Generator(device=DEV).manual_seed(seed * 7 + 1)
    noise = torch.randn((c["M"], 2), generator=gen, device=DEV, dtype=torch.float64)
    y += torch.view_as_complex(noise) * (tau / math.sqrt(2.0))
    if g["d"] is not None:
        d = torch.from_numpy(g["d"]).to(DEV)
        y *= d
        tau *= float(d.square().mean().sqrt())
    return y.to(torch.complex64), tau, sky


def _facets(c, seed):
    n, f = c["n"], c["facets"]
    rng = np.random.default_rng([seed, 13])
    out = []
    for _ in range(2):
        wd = np.full(f, n / f) if c.get("even") else n * (q := rng.uniform(768, 1280, f)) / q.sum()
        cuts = np.rint(np.concatenate([[0.0], np.cumsum(wd)])).astype(int)
        out.append(np.diff(cuts).astype(np.int32))
    return out


def _loop_inputs(c, seed):
    g = _geometry(c, seed)
    y, tau, sky = _data(c, g, seed)
    gamma, t = 1.98 / g["L"], tau / math.sqrt(2.0 * g["L"])
    s = dict(g=g, y=y, gamma=gamma, t=t, L=g["L"], alpha=1.0)
    if c["kind"] == "learned":
        s["params"], meta = load_weights(WEIGHTS)
        s["alpha"] = max(2.0, alpha_for_denoiser(tau, g["L"], float(meta["sigma"])))
    if c["kind"] in ("grad", "dirty"):  # an iterate on its way to the sky: half of it, with the noise of an early image
        gen = torch.Generator(device=DEV).manual_seed(seed * 7 + 2)
        x = _sky_image(c["n"], sky)
        s["x"] = (0.5 * x + 1e-3 * torch.randn(x.shape, generator=gen, device=DEV)).contiguous()
    return s


def _net(seed, last):
    """He-normal weights, small random biases, a small last layer: a network early in its training."""
    rng = np.random.default_rng([seed, 14])
    out = []
    for i, (co, ci) in enumerate([(64, 1)] + [(64, 64)] * 6 + [(1, 64)]):
        sd = math.sqrt(2.0 / (9 * ci)) * (last if i == 7 else 1.0)
        out.append((rng.normal(0.0, sd, (co, ci, 3, 3)), rng.normal(0.0, 0.01, co)))
    return out


def _batch(c, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed * 7 + 3)
    rng = np.random.default_rng([seed, 15])
    u = torch.stack([_sky_image(c["size"], _sky(c["size"], rng)) for _ in range(c["batch"])])
    u /= u.amax((1, 2), keepdim=True)
    return [u] + [torch.randn(u.shape, generator=gen, device=DEV) for _ in range(2)]


def _noisy_image(c, seed, sigma):
    gen = torch.Generator(device=DEV).manual_seed(seed * 7 + 4)
    x = _sky_image(c["n"], _sky(c["n"], np.random.default_rng([seed, 16])))
    x = x / x.max()
    return (x + sigma * torch.randn(x.shape, generator=gen, device=DEV)).contiguous()


SIGMA_TRAIN, SARA_SIGMA, FNE_LAMBDA, FNE_EPS = 0.05, 1e-3, 10.0, 0.05


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "cnn":
        params, meta = load_weights(WEIGHTS)
        fr, fc = _facets(c, seed)
        return dict(c=c, z=_noisy_image(c, seed, float(meta["sigma"])),
                    den=pnp.CnnDenoiser(params, c["n"], facet_rows=fr, facet_cols=fc, halo=32))
    if c["kind"] == "sara":
        return dict(c=c, z=_noisy_image(c, seed, SARA_SIGMA),
                    den=pnp.SaraDenoiser(c["n"], SARA_SIGMA, SARA_SIGMA, c["prox"]))
    if c["kind"] in ("train", "train_fne"):
        u, noise, v0 = _batch(c, seed)
        return dict(c=c, u=u, noise=noise, v0=v0, tr=pnp.CnnTrainer(_net(seed, 0.1), c["batch"], c["size"]))
    s = dict(c=c, **_loop_inputs(c, seed))
    g = s.pop("g")
    s["plan"] = pnp.Plan(c["n"], c["K"], g["omega"], g["w"], g["dl"], g["Jr"], J=g["J"], weight_dtype=c["weights"],
                         block=g["block"], nblocks=c["blocks"], stack=g["stack"], w_centres=g["centres"],
                         row_scale=g["d"])
    if c["holo"]:
        s["plan"].set_holographic(True)
    if c["kind"] == "fb":
        s["den"] = pnp.HaarDenoiser(s["t"])
    if c["kind"] == "learned":
        fr, fc = _facets(c, seed)
        s["den"] = pnp.CnnDenoiser(s["params"], c["n"], facet_rows=fr, facet_cols=fc, halo=32)
    return s


def run(state):
    c = state["c"]
    kind = c["kind"]
    if kind in ("cnn", "sara"):
        return state["den"].denoise(state["z"])
    if kind == "train":
        loss = state["tr"].step(state["u"], state["noise"], SIGMA_TRAIN, update=False, want_loss=True)
        return {"loss": loss, "grads": state["tr"].read(weights=False, grads=True, clear_grads=True)[1]}
    if kind == "train_fne":
        loss, pen = state["tr"].step_fne(state["u"], state["noise"], SIGMA_TRAIN, state["v0"], c["iters"], FNE_LAMBDA,
                                         FNE_EPS, update=False, want_values=True)
        return {"loss": loss, "penalty": pen,
                "grads": state["tr"].read(weights=False, grads=True, clear_grads=True)[1]}
    if kind == "grad":
        return state["plan"].grad_step(state["x"], state["y"], state["gamma"])
    if kind == "dirty":
        return {"vis": state["plan"].phi_forward(state["x"]), "dirty": state["plan"].phi_adjoint(state["y"])}
    x, st = state["plan"].fb_run(state["den"], state["y"], gamma=state["gamma"], L=state["L"],
                                 max_iter=c["iters"], alpha=state["alpha"])
    return {"x": x, "rel_change": st.rel_change, "x_norm": st.x_norm}


# ------------------------------------------------------------------------------------------------ work
def _mean_taps(c):
    """Mean (J_m^2, J_m) of a row: the supports take a quarter of the rows each."""
    s = [int(v) for v in c["supports"].split(",")]
    return sum(v * v for v in s) / len(s), sum(s) / len(s)


def work(case):
    c = dict(case)
    if c["kind"] == "cnn":
        px = c["n"] ** 2
        return {"bytes": 8 * px, "flops": CNN_FLOP_PER_PX * px}
    if c["kind"] == "sara":  # per dual iteration: read and write the 9 dual images, read the 9 weights and z
        px = c["n"] ** 2
        return {"bytes": px * 4 * (c["prox"] * 28 + 10), "flops": px * c["prox"] * 2 * 9 * 2 * 2 * 9 * 4 // 3}
    if c["kind"] in ("train", "train_fne"):
        px = c["batch"] * c["size"] ** 2
        passes = 3 + (2 * c["iters"] + 3 if c["kind"] == "train_fne" else 0)
        return {"bytes": 12 * px + 4 * 223_041, "flops": passes * CNN_FLOP_PER_PX * px}
    n2, M, (taps, sup) = c["n"] ** 2, c["M"], _mean_taps(c)
    wb = 8 if c["weights"] == "c64" else 4
    fft = 4 * 2.5 * c["n"] * c["K"] * math.log2(c["K"]) * c["stacks"]
    if c["kind"] == "dirty":  # the two axes' weights of a row (G is separable), visibilities, images
        return {"bytes": 2 * (M * (2 * sup * 8 + 8) + 4 * n2), "flops": 16 * M * taps + 2 * fft}
    if c["holo"]:
        S = 2 * max(int(v) for v in c["supports"].split(",")) - 1
        per = {"bytes": S * S * c["K"] ** 2 * 8 + 8 * n2, "flops": 8 * S * S * c["K"] ** 2 + 2 * fft}
    else:
        per = {"bytes": M * (2 * sup * wb + 8) + 8 * n2, "flops": 16 * M * taps + 2 * fft}
    if c["kind"] == "learned":
        per = {"bytes": per["bytes"] + 8 * n2, "flops": per["flops"] + CNN_FLOP_PER_PX * n2}
    return {k: v * c["iters"] for k, v in per.items()}


# ------------------------------------------------------------------------------------------------ 64 bits
class _Operator:
    """Phi = D G F Z in double precision: KB rows, each convolved with its row's w-kernel, per w-stack."""

    def __init__(self, c, g):
        self.n, self.K, self.g = c["n"], c["K"], g
        n, K, J = self.n, self.K, g["J"]
        s = K / n
        self.beta = beta = math.pi * math.sqrt((J / s) ** 2 * (s - 0.5) ** 2 - 0.8)
        p = np.arange(n) - n // 2
        r = np.sqrt((beta ** 2 - (np.pi * J * p / K) ** 2).astype(complex))
        self.cinv = torch.from_numpy(np.real(r / (J * np.sinh(r)))).to(DEV)
        self.pos = torch.from_numpy(p % K).to(DEV)
        wres = g["w"] - (0.0 if g["stack"] is None else g["centres"][g["stack"]])
        a = torch.from_numpy(wres * g["dl"] ** 2).to(DEV)
        Jr = torch.full((c["M"],), J, device=DEV) if g["Jr"] is None else torch.from_numpy(g["Jr"]).to(DEV).long()
        st = torch.zeros(c["M"], dtype=torch.long, device=DEV) if g["stack"] is None else torch.from_numpy(g["stack"]).to(DEV).long()
        om = torch.from_numpy(g["omega"]).to(DEV) * (K / (2 * math.pi))
        d = torch.ones(c["M"], dtype=torch.float64, device=DEV) if g["d"] is None else torch.from_numpy(g["d"]).to(DEV)
        cheb = self._wkernel(a) if g["dl"] else None
        self.parts = []  # per (stack, support): rows, first taps per axis, the two axes' weights
        for k in range(c["stacks"]):
            for Jm in torch.unique(Jr).tolist():
                rows = torch.nonzero((st == k) & (Jr == Jm)).ravel()
                for q in rows.split(1 << 18):
                    if q.numel():
                        s0 = torch.floor(om[q] - 0.5 * Jm).long() + 1
                        f = [self._row(om[q, ax] - s0[:, ax], Jm, a[q], cheb) for ax in (0, 1)]
                        f[0] = f[0] * d[q, None]
                        self.parts.append((k, Jm, q, s0, f))
        self.chirp = None
        if c["stacks"] > 1:
            q2 = torch.from_numpy((p.astype(float)) ** 2).to(DEV)
            self.chirp = [torch.polar(torch.ones_like(q2), math.pi * w * g["dl"] ** 2 * q2) for w in g["centres"]]
        self.stacks, self.M = c["stacks"], c["M"]

    def _wkernel(self, a):
        """Chebyshev coefficients in a of w_hat[d] = K^-1 sum_p exp(i pi a q(p)) cos(2 pi d p / K), d = -16..16."""
        n, K, N = self.n, self.K, 96
        self.amax = amax = max(float(a.abs().max()), 1e-300)
        p = torch.arange(K, device=DEV, dtype=torch.float64) - K // 2
        h = n / 2.0
        u = (p.abs() - h).clamp(min=0) / (K / 2 - h)
        q = torch.where(p.abs() <= h, p * p, h * h + n * (K / 2 - h) * (u + u * u / 2 - u ** 4 + 0.4 * u ** 5))
        nodes = torch.cos(math.pi * (torch.arange(N, device=DEV, dtype=torch.float64) + 0.5) / N)
        ph = math.pi * amax * nodes[:, None] * q[None]
        dd = torch.arange(-16, 17, device=DEV, dtype=torch.float64)
        vals = torch.polar(torch.ones_like(ph), ph) @ torch.cos(2 * math.pi / K * p[:, None] * dd[None]).to(torch.complex128) / K
        T = torch.cos(torch.arange(N, device=DEV, dtype=torch.float64)[:, None] * torch.acos(nodes)[None])
        co = (2.0 / N) * T.to(torch.complex128) @ vals
        co[0] *= 0.5
        return co

    def _row(self, t0, Jm, a, cheb):
        def psi(t):
            z = 1.0 - (2.0 * t / self.g["J"]) ** 2
            return torch.where(z >= 0, torch.special.i0(self.beta * torch.sqrt(z.clamp(min=0))), torch.zeros_like(z))
        J = self.g["J"]
        sl = torch.arange(Jm, device=DEV)
        if cheb is None:
            return psi(t0[:, None] - sl).to(torch.complex128)
        x = (a / self.amax).clamp(-1, 1)[:, None].to(torch.complex128)
        b1 = b2 = torch.zeros((a.numel(), 33), dtype=torch.complex128, device=DEV)
        for k in range(cheb.shape[0] - 1, 0, -1):
            b1, b2 = cheb[k] + 2 * x * b1 - b2, b1
        wh = cheb[0] + x * b1 - b2
        wh = torch.where((a == 0)[:, None], (torch.arange(-16, 17, device=DEV) == 0).to(torch.complex128)[None], wh)
        emin = torch.ceil(-t0 - 0.5 * J).long()
        out = torch.zeros((a.numel(), Jm), dtype=torch.complex128, device=DEV)
        for i in range(J + 1):
            e = emin + i
            idx = (e[:, None] + sl[None] + 16)
            ok = (idx >= 0) & (idx <= 32)
            out += psi(t0 + e)[:, None] * torch.gather(wh, 1, idx.clamp(0, 32)) * ok
        return out

    def _taps(self, s0, Jm):
        sl = torch.arange(Jm, device=DEV)
        return ((s0[:, 0, None] + sl) % self.K), ((s0[:, 1, None] + sl) % self.K)

    def forward(self, x):
        y = torch.empty(self.M, dtype=torch.complex128, device=DEV)
        for k in range(self.stacks):
            z = (x * self.cinv[:, None] * self.cinv[None]).to(torch.complex128)
            if self.chirp:
                z = z * self.chirp[k][:, None] * self.chirp[k][None]
            X = torch.zeros((self.K, self.K), dtype=torch.complex128, device=DEV)
            X[self.pos[:, None], self.pos[None]] = z
            X = torch.fft.fft2(X).ravel()
            for q, Jm, rows, s0, f in self.parts:
                if q == k:
                    k0, k1 = self._taps(s0, Jm)
                    acc = torch.zeros(rows.numel(), dtype=torch.complex128, device=DEV)
                    for i in range(Jm):
                        acc += f[0][:, i] * (f[1] * X[k0[:, i, None] * self.K + k1]).sum(1)
                    y[rows] = acc
        return y

    def adjoint(self, y):
        out = torch.zeros((self.n, self.n), dtype=torch.float64, device=DEV)
        for k in range(self.stacks):
            G = torch.zeros((self.K * self.K, 2), dtype=torch.float64, device=DEV)
            for q, Jm, rows, s0, f in self.parts:
                if q == k:
                    k0, k1 = self._taps(s0, Jm)
                    for i in range(Jm):
                        v = (f[0][:, i].conj() * y[rows])[:, None] * f[1].conj()
                        G.index_add_(0, (k0[:, i, None] * self.K + k1).ravel(), torch.view_as_real(v).reshape(-1, 2))
            z = torch.fft.ifft2(torch.view_as_complex(G).view(self.K, self.K), norm="forward")[self.pos[:, None], self.pos[None]]
            if self.chirp:
                z = z * (self.chirp[k][:, None] * self.chirp[k][None]).conj()
            out += z.real * self.cinv[:, None] * self.cinv[None]
        return out


def _haar(z, t):
    a, b, c, d = z[0::2, 0::2], z[0::2, 1::2], z[1::2, 0::2], z[1::2, 1::2]
    s = [0.5 * (a + b + c + d), 0.5 * (a - b + c - d), 0.5 * (a + b - c - d), 0.5 * (a - b - c + d)]
    s = [torch.sign(v) * (v.abs() - t).clamp(min=0) for v in s]
    o = torch.empty_like(z)
    o[0::2, 0::2] = 0.5 * (s[0] + s[1] + s[2] + s[3])
    o[0::2, 1::2] = 0.5 * (s[0] - s[1] + s[2] - s[3])
    o[1::2, 0::2] = 0.5 * (s[0] + s[1] - s[2] - s[3])
    o[1::2, 1::2] = 0.5 * (s[0] - s[1] - s[2] + s[3])
    return o.clamp(min=0)


def _conv(h, W, b):
    """3 x 3 'same' convolution of h (channels, rows, columns) as nine products, in bands of rows."""
    H, Wd = h.shape[1:]
    hp = torch.nn.functional.pad(h, (1, 1, 1, 1))
    out = torch.empty((W.shape[0], H, Wd), dtype=torch.float64, device=DEV)
    for r in range(0, H, 256):
        k = min(256, H - r)
        acc = b[:, None].expand(-1, k * Wd).clone()
        for t in range(9):
            acc += W[:, :, t // 3, t % 3] @ hp[:, r + t // 3:r + t // 3 + k, t % 3:t % 3 + Wd].reshape(h.shape[0], -1)
        out[:, r:r + k] = acc.view(-1, k, Wd)
    return out


def _cnn(z, params):
    """max(0, z - N(z)); facets with a halo of at least 8 pixels give the whole image's result."""
    h = z[None]
    for i, (W, b) in enumerate(params):
        h = _conv(h, torch.from_numpy(W).to(DEV), torch.from_numpy(b).to(DEV))
        if i < 7:
            h.clamp_(min=0)
    return (z - h[0]).clamp(min=0)


def _daubechies(N):
    Q = np.zeros(2 * N - 1)
    for k in range(N):
        t = np.array([1.0])
        for _ in range(k):
            t = np.polymul(t, [-0.25, 0.5, -0.25])
        t = np.concatenate([t, np.zeros(N - 1 - k)])
        Q[-t.size:] += math.comb(N - 1 + k, k) * t
    h = np.array([1.0])
    if N > 1:
        r = np.roots(Q)
        for _ in range(3):
            r = r - np.polyval(Q, r) / np.polyval(np.polyder(Q), r)
        h = np.real(np.poly(r[np.abs(r) < 1]))
    for _ in range(N):
        h = np.polymul(h, [1.0, 1.0])
    return h * (math.sqrt(2.0) / h.sum())


def _analyse(x, f, levels=4):
    hp = [(-1) ** k * f[len(f) - 1 - k] for k in range(len(f))]
    c, m = x.clone(), x.shape[0]
    for _ in range(levels):
        b = c[:m, :m]
        for ax in (0, 1):
            step = (slice(None, None, 2), slice(None)) if ax == 0 else (slice(None), slice(None, None, 2))
            b = torch.cat([sum(float(v) * torch.roll(b, -k, ax)[step] for k, v in enumerate(q)) for q in (f, hp)], ax)
        c[:m, :m] = b
        m //= 2
    return c


def _synthesise(c, f, levels=4):
    hp = [(-1) ** k * f[len(f) - 1 - k] for k in range(len(f))]
    x, m = c.clone(), c.shape[0] >> (levels - 1)
    for _ in range(levels):
        b = x[:m, :m]
        for ax in (1, 0):
            out = 0.0
            for half, q in zip(b.chunk(2, ax), (f, hp)):
                up = torch.zeros_like(b)
                up[(slice(None, None, 2), slice(None)) if ax == 0 else (slice(None), slice(None, None, 2))] = half
                out = out + sum(float(v) * torch.roll(up, k, ax) for k, v in enumerate(q))
            b = out
        x[:m, :m] = b
        m *= 2
    return x


def _sara(z, t, iters):
    fl = [_daubechies(N) for N in range(1, 9)]
    u = [torch.zeros_like(z) for _ in range(9)]

    def primal():
        return (z - (u[0] + sum(_synthesise(u[b], fl[b - 1]) for b in range(1, 9))) / 3.0).clamp(min=0)
    x = primal()
    for _ in range(iters):
        u = [(u[b] + (x if b == 0 else _analyse(x, fl[b - 1])) / 3.0).clamp(-t, t) for b in range(9)]
        x = primal()
    return x


def _train_exact(c, seed):
    """Loss (and penalty) and flat gradients of the training step, the network unrounded."""
    u, noise, v0 = (t.double() for t in _batch(c, seed))
    z = (u + SIGMA_TRAIN * noise)[:, None]
    flat = [torch.from_numpy(a).to(DEV).requires_grad_() for p in _net(seed, 0.1) for a in p]
    Ws, bs = flat[0::2], flat[1::2]
    conv = torch.nn.functional.conv2d
    h, masks = z, []
    for i in range(8):
        h = conv(h, Ws[i], bs[i], padding=1)
        if i < 7:
            masks.append((h > 0).double().detach())
            h = h * masks[i]
    loss = (z - h - u[:, None]).abs().mean()
    grads = list(torch.autograd.grad(loss, flat))
    out = {"loss": float(loss.detach())}
    if c["kind"] == "train_fne":
        def J(v):
            t = v
            for i in range(8):
                t = conv(t, Ws[i], padding=1)
                t = t * masks[i] if i < 7 else t
            return v - 2.0 * t

        def unit(v):
            return v / v.square().sum((1, 2, 3), keepdim=True).sqrt()
        v = unit(v0[:, None])
        for _ in range(c["iters"]):
            v = v.detach().requires_grad_()
            r = J(v)
            v = unit(torch.autograd.grad(r, v, r.detach())[0])
        pen = (FNE_LAMBDA / c["batch"]) * J(v.detach()).square().sum((1, 2, 3)).clamp(min=1 - FNE_EPS).sum()
        out["penalty"] = float(pen.detach())
        more = torch.autograd.grad(pen, Ws)
        for i in range(8):
            grads[2 * i] = grads[2 * i] + more[i]
    return out | {"grads": torch.cat([q.reshape(-1) for q in grads]).cpu().numpy()}


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "cnn":
        params, meta = load_weights(WEIGHTS)
        return _cnn(_noisy_image(c, seed, float(meta["sigma"])).double(), params)
    if c["kind"] == "sara":
        return _sara(_noisy_image(c, seed, SARA_SIGMA).double(), float(np.float32(SARA_SIGMA)), c["prox"])
    if c["kind"] in ("train", "train_fne"):
        return _train_exact(c, seed)
    s = _loop_inputs(c, seed)
    op, y = _Operator(c, s["g"]), s["y"].to(torch.complex128) / s["alpha"]
    if c["kind"] == "grad":
        x = s["x"].double()
        return x - s["gamma"] * op.adjoint(op.forward(x) - y)
    if c["kind"] == "dirty":
        return {"vis": op.forward(s["x"].double()), "dirty": op.adjoint(y)}
    x = torch.zeros((c["n"], c["n"]), dtype=torch.float64, device=DEV)
    for _ in range(c["iters"]):
        prev, z = x, x - s["gamma"] * op.adjoint(op.forward(x) - y)
        x = _haar(z, s["t"]) if c["kind"] == "fb" else _cnn(z, s["params"])
    xn = float(x.norm())
    return {"x": x * s["alpha"], "rel_change": float((x - prev).norm()) / xn if xn else 0.0, "x_norm": xn}
