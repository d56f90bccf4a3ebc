"""The calls whose speed is followed: reconstructions over the range of meshes and catalogues, and the
layers a program calls by themselves (the shift, the survey front end, the network, the
finite-difference method).

A case is a dict of plain values; its "kind" names the call:
  recon     deposit -> smooth -> iterate -> shift of the galaxies and randoms, one handle
  batch     several mocks of mixed mesh sides through batch_run
  shift     one catalogue moved along a solved displacement, shifted positions included
  frontend  n(r), FKP weights and the weighted nearest-grid-point deposit of galaxies and randoms
  fd        the finite-difference solve after smoothing
  infer     the warm-start network's forward pass
  train     one training step of it (forward, loss, gradients, AdamW)
Inputs are drawn on the GPU from the seed with the workloads' own generator (mocks.batch_mock_device).
`exact` computes the same values with plain torch in float64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1504_02591_gb300 import binding as B
from paper_1504_02591_gb300 import mocks, warmstart

STARTS = {"plain": B.START_PLAIN, "approx1": B.START_APPROX1, "approx2": B.START_FFTA, "learned": B.START_FFTA}


def _recon(name, n, L, shell, n_gal, ratio, **kw):
    c = dict(kind="recon", n=n, L=float(L), shell=shell, n_gal=n_gal, ratio=ratio, b=1.85, f=0.74, R=15.0,
             los="radial", lognormal=False, dtype="f64", start="approx2", tol=1e-6, max_iter=80, sorted=False)
    c.update(kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest reconstruction: a quick look at one small box, float32 positions, flat-sky line
        # of sight, logarithmic density, no correction in the start; launches and latency count
        _recon("box32", 32, 500.0, False, 20_000, 0, b=2.0, los="fixed", lognormal=True, dtype="f32",
               start="plain", tol=0.0, max_iter=4),
        # the small periodic box with randoms (six updates): the everyday interactive call
        _recon("box64", 64, 1000.0, False, 200_000, 10, b=2.0, tol=0.0, max_iter=6),
        # one mock survey of a covariance set on the small mesh, to convergence
        _recon("shell256", 256, 1751.0, True, 403_117, 37, b=2.1, f=0.7),
        # one periodic mock on the radix-3 mesh, to convergence
        _recon("box384", 384, 2626.6, False, 751_333, 0, b=1.6, f=0.78),
        # the survey workload with the learned start: one brick sort per catalogue, reused by the shift
        _recon("survey512", 512, 3500.0, True, 600_000, 50, start="learned", sorted=True),
        # the large periodic run: 1e8 particles, six updates
        _recon("box1024", 1024, 2500.0, False, 100_000_000, 0, b=1.0, R=10.0, tol=0.0, max_iter=6, sorted=True),
        # a few mocks of a covariance set, mixed mesh sides, surveys and boxes, in one call
        dict(name="batch", kind="batch", count=6, n_lo=256, n_hi=384, gal_lo=200_000, gal_hi=1_000_000, ratio=30),
        # another large catalogue moved along a solved field (float32 positions, positions out)
        dict(name="shift", kind="shift", n=256, L=1751.0, count=10_000_019, dtype="f32", galaxy=True, periodic=True),
        # the survey's weights and binned densities from raw catalogues, as the paper prepares them
        dict(name="frontend", kind="frontend", n=256, L=3500.0, n_gal=600_000, ratio=50, nbins=50, dtype="f64"),
        # the paper's comparison method on a mid-size box
        dict(name="fd", kind="fd", n=128, L=1000.0, n_gal=400_000, f=0.74, tol=1e-5, los="radial"),
        # the network at the survey workload's coarse mesh: one forward pass
        dict(name="infer", kind="infer", n=128, c1=8, bf16=True),
        # one step of its training at the same mesh
        dict(name="train", kind="train", n=128, c1=8, bf16=True),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["recon"] * 6 + ["batch", "shift", "shift", "frontend", "fd", "infer", "train"])
    if kind == "recon":
        n = rng.choice([32, 48, 64, 96, 128, 256, 384, 512, 1024])
        shell = n < 1024 and rng.random() < 0.5
        cells = n ** 3
        n_gal = _logint(rng, max(5_000, cells // 2000), max(20_000, min(cells // 4, 40_000_000 if n == 1024 else 4_000_000)))
        if shell:
            n_gal = min(n_gal, 700_000)
        ratio = rng.randint(10, 50) if shell else rng.choice([0, 0, rng.randint(3, 12)])
        ratio = min(ratio, 30_000_000 // n_gal)
        if shell:
            ratio = max(ratio, 10)
        fixed = rng.random() < 0.5
        return _recon(None, n, round(n * rng.uniform(6.0, 16.0), 1), shell, n_gal, ratio,
                      b=round(rng.uniform(1.0 if not shell else 1.5, 2.5), 3), f=round(rng.uniform(0.5, 0.85), 3),
                      R=round(rng.uniform(8.0, 20.0), 2), los="fixed" if not shell and rng.random() < 0.3 else "radial",
                      lognormal=rng.random() < 0.2, dtype=rng.choice(["f64", "f64", "f32"]),
                      start=rng.choice(["plain", "approx1", "approx2", "approx2"]), tol=0.0 if fixed or n == 1024 else 1e-6,
                      max_iter=rng.randint(2, 6) if fixed or n == 1024 else 80, sorted=rng.random() < 0.5)
    if kind == "batch":
        hi = rng.choice([64, 128, 256, 384, 512])
        return dict(kind="batch", count=rng.randint(2, 6), n_lo=32, n_hi=hi, gal_lo=20_000, gal_hi=_logint(rng, 50_000, 600_000),
                    ratio=rng.randint(10, 40))
    if kind == "shift":
        return dict(kind="shift", n=rng.choice([64, 128, 256, 384, 512]), L=round(rng.uniform(500.0, 3500.0), 1),
                    count=_logint(rng, 10_000, 30_000_000), dtype=rng.choice(["f32", "f64"]), galaxy=rng.random() < 0.5,
                    periodic=rng.random() < 0.5)
    if kind == "frontend":
        return dict(kind="frontend", n=rng.choice([64, 128, 256, 384]), L=round(rng.uniform(1500.0, 3500.0), 1),
                    n_gal=_logint(rng, 20_000, 600_000), ratio=rng.randint(10, 50), nbins=rng.randint(10, 200),
                    dtype=rng.choice(["f64", "f64", "f32"]))
    if kind == "fd":
        n = rng.choice([32, 48, 64, 96, 128])
        return dict(kind="fd", n=n, L=round(n * rng.uniform(7.0, 15.0), 1), n_gal=_logint(rng, 20_000, 500_000),
                    f=round(rng.uniform(0.3, 0.8), 3), tol=1e-5, los=rng.choice(["radial", "fixed"]))
    n = rng.choice([16, 32, 40, 64, 96, 128, 160] + ([192, 256] if kind == "infer" else []))
    return dict(kind=kind, n=n, c1=8 if n > 128 else rng.choice([8, 16]), bf16=rng.random() < 0.7 or kind == "infer")


# ---- inputs -------------------------------------------------------------------------------------
def _cast(pos, dtype):
    return pos if pos is None or dtype == "f64" else pos.to(torch.float32)


def _periodic_f32(pos, L):
    """float32 positions stay inside [0, L) (rounding up to L stands for 0)."""
    if pos is not None and pos.dtype == torch.float32:
        pos[pos >= L] = 0.0
    return pos


def _mock(c, seed):
    """(params, galaxies, randoms) of a recon case."""
    m = mocks.batch_mock_device(c["n"], c["n_gal"], max(c["ratio"], 1), c["b"], c["f"], c["shell"], seed, L=c["L"])
    p = dict(m["params"], R=c["R"], lognormal=c["lognormal"])
    ran = m["ran"]
    if not c["shell"] and c["ratio"]:
        g = torch.Generator(device="cuda").manual_seed(seed + 1)
        ran = torch.rand((c["n_gal"] * c["ratio"], 3), generator=g, device="cuda", dtype=torch.float64) * c["L"]
        p["uniform"] = False
    if c["los"] == "fixed":
        p.update(los_mode=B.LOS_FIXED, observer=(0.8, -0.36, 0.48))
    gal, ran = _periodic_f32(_cast(m["gal"], c["dtype"]), c["L"]), _periodic_f32(_cast(ran, c["dtype"]), c["L"])
    return p, gal, ran


def _handle(p):
    return B.Recon(p["n"], p["L"], p["b"], p["f"], p["R"], p["observer"], p["los_mode"], p["periodic"], p["mask_frac"],
                   p["lognormal"], p["uniform"])


def _batch_mocks(c, seed):
    rng = np.random.default_rng(seed)
    sides = [n for n in (32, 48, 64, 96, 128, 256, 384, 512) if c["n_lo"] <= n <= c["n_hi"]]
    out = []
    for i in range(c["count"]):
        n_gal = c["gal_lo"] + int((c["gal_hi"] - c["gal_lo"]) * (i * 0.618 % 1.0))   # sizes are the case's, not the seed's
        out.append(mocks.batch_mock_device(sides[i % len(sides)], n_gal, c["ratio"], float(rng.uniform(1.5, 2.5)),
                                           float(rng.uniform(0.6, 0.8)), i % 2 == 0, seed + 10 * i))
    return out


def _shift_inputs(c, seed):
    """A box's params and galaxies for the solve, and the catalogue to move (uniform in the box)."""
    m = mocks.batch_mock_device(c["n"], max(20_000, c["n"] ** 3 // 40), 1, 1.8, 0.75, False, seed, L=c["L"])
    p = dict(m["params"], periodic=c["periodic"])
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    pos = torch.rand((c["count"], 3), generator=g, device="cuda", dtype=torch.float64) * c["L"]
    return p, m["gal"], _periodic_f32(_cast(pos, c["dtype"]), c["L"])


def _shells(c):
    s = c["L"] / 3500.0
    return 1100.0 * s, 1800.0 * s, math.pi   # r_min, r_max, a quarter of the sky in steradians


def _fd_inputs(c, seed):
    m = mocks.batch_mock_device(c["n"], c["n_gal"], 1, 2.0, c["f"], False, seed, L=c["L"])
    p = dict(m["params"])
    if c["los"] == "fixed":
        p.update(los_mode=B.LOS_FIXED, observer=(0.6, 0.0, 0.8))
    return p, m["gal"]


def _net_inputs(c, seed):
    """Flat parameters (He-scaled draws, small biases), input features and target.  The features look
    like the solver's: a smooth overdensity, the line of sight, and a displacement of a few Mpc/h."""
    specs, c1 = [], c["c1"]
    for ci, co, taps in [(5, c1, 27), (c1, c1, 27), (c1, 2 * c1, 27), (2 * c1, 2 * c1, 27), (2 * c1, 4 * c1, 27),
                         (4 * c1, 4 * c1, 27), (6 * c1, 2 * c1, 27), (2 * c1, 2 * c1, 27), (3 * c1, c1, 27), (c1, c1, 27),
                         (c1, 1, 1)]:
        specs.append((ci, co, taps))
    rng = np.random.default_rng(seed)
    flat = []
    for ci, co, taps in specs:
        flat.append(rng.standard_normal(taps * ci * co).astype(np.float32) * np.float32(math.sqrt(2.0 / (taps * ci))))
        flat.append(rng.standard_normal(co).astype(np.float32) * np.float32(0.05))
    n = c["n"]
    F = mocks._field_device(n, 27.0 * n, torch.Generator(device="cuda").manual_seed(seed), "cuda")
    a = (torch.arange(n, device="cuda", dtype=torch.float32) + 0.5) / n
    d = torch.stack(torch.meshgrid(a, a - 0.5, a - 0.5, indexing="ij"), -1)
    r = d / torch.linalg.norm(d, dim=-1, keepdim=True)
    u = (F[1:].permute(1, 2, 3, 0) * r).sum(-1)
    x = torch.cat([F[0][..., None].clamp(-1.0, 5.0), r, u[..., None]], -1).contiguous()
    return np.concatenate(flat), specs, x, (u * 1.15 + 0.3 * F[0]).contiguous()


# ---- states and passes --------------------------------------------------------------------------
def prepare(case, seed):
    c, k = case, case["kind"]
    if k == "recon":
        p, gal, ran = _mock(c, seed)
        h = _handle(p)
        if c["sorted"]:
            h.set_option(B.OPT_DEPOSIT_PATH, B.PATH_SORTED)
            h.set_option(B.OPT_REUSE_SORT, 1)
        net, level = warmstart.load(warmstart.default_weights_path()) if c["start"] == "learned" else (None, 0)
        return dict(c=c, h=h, gal=gal, ran=ran, net=net, level=level)
    if k == "batch":
        return dict(c=c, mocks=_batch_mocks(c, seed))
    if k == "shift":
        p, gal, pos = _shift_inputs(c, seed)
        h = _handle(p)
        h.run(gal, None, B.START_FFTA, 0.0, 3)
        return dict(c=c, h=h, pos=pos)
    if k == "frontend":
        m = mocks.batch_mock_device(c["n"], c["n_gal"], c["ratio"], 1.85, 0.74, True, seed, L=c["L"])
        h = _handle(m["params"])
        h.set_option(B.OPT_ASSIGN, B.ASSIGN_NGP)
        return dict(c=c, h=h, gal=_cast(m["gal"], c["dtype"]), ran=_cast(m["ran"], c["dtype"]))
    if k == "fd":
        p, gal = _fd_inputs(c, seed)
        h = _handle(p)
        h.deposit(gal)
        h.smooth()
        return dict(c=c, h=h)
    flat, _, x, t = _net_inputs(c, seed)
    net = B.UNet(c1=c["c1"], bf16=c["bf16"])
    net.set_params(flat)
    return dict(c=c, net=net, x=x, t=t)


def run(state):
    c, k = state["c"], state["c"]["kind"]
    if k == "recon":
        h, gal, ran = state["h"], state["gal"], state["ran"]
        h.deposit(gal, None, ran, None)
        h.smooth()
        if state["net"] is not None:
            n_it, _, _ = warmstart.warm_iterate(h, state["net"], state["level"], c["tol"], c["max_iter"])
        else:
            n_it, _, _ = h.iterate(STARTS[c["start"]], c["tol"], c["max_iter"])
        out = dict(n_iter=n_it, shift_gal=h.shift(gal, True))
        if ran is not None:
            out["shift_ran"] = h.shift(ran, False)
        out["psi"] = h.get_psi()
        return out
    if k == "batch":
        _, res = B.batch_run(state["mocks"], start=B.START_FFTA, tol=1e-6, max_iter=80)
        return [[r["n_iter"], r["shift_gal"], r["shift_ran"]] for r in res]
    if k == "shift":
        shift, pos = state["h"].shift(state["pos"], c["galaxy"], want_pos=True)
        return dict(shift=shift, pos=pos)
    if k == "frontend":
        h, gal, ran = state["h"], state["gal"], state["ran"]
        rmin, rmax, area = _shells(c)
        nbar = h.radial_nbar(gal, c["nbins"], rmin, rmax, area)
        wg, wr = h.fkp_weights(gal, nbar, rmin, rmax), h.fkp_weights(ran, nbar, rmin, rmax)
        h.deposit(gal, wg, ran, wr)
        return dict(nbar=nbar, w_gal=wg, w_ran=wr, rho_gal=h.get_field(B.FIELD_RHO_G), rho_ran=h.get_field(B.FIELD_RHO_R))
    if k == "fd":
        return state["h"].fd_solve(c["tol"], 200)[0]
    net, x = state["net"], state["x"]
    if k == "infer":
        return net.forward(x)
    loss = net.backward(x, state["t"])
    net.adamw(1e-4)
    return dict(loss=torch.tensor(loss, dtype=torch.float32), grads=net.get_grads(), params=net.get_params())


# ---- the least work of a pass -------------------------------------------------------------------
def _recon_work(n, n_gal, n_ran, es, updates):
    """Catalogues read and shifts written once, one real density field per catalogue, the displacement
    written once; transforms: one 3-D FFT of delta, and per update two scalar fields each way (the
    least that carries the vector through), 2.5 N^3 log2 N^3 operations a real transform."""
    cells, particles = n ** 3, n_gal + n_ran
    fft = 2.5 * cells * 3 * math.log2(n)
    return dict(bytes=particles * (3 * es + 12) + cells * 4 * (1 + (n_ran > 0)) * 2 + cells * 4 * 3
                + updates * 2 * cells * 8.0, flops=fft * (1 + 6 * updates) + particles * 100.0)


def _net_flops(n, c1):
    v = n ** 3
    pairs = (5 * c1 + c1 * c1) + (3 * c1 * c1 + c1 * c1), (2 * c1 * c1 + 4 * c1 * c1 + 12 * c1 * c1 + 4 * c1 * c1), \
            (8 * c1 * c1 + 16 * c1 * c1)
    return 54.0 * (pairs[0] * v + pairs[1] * v / 8 + pairs[2] * v / 64)


def work(case):
    c, k = case, case["kind"]
    if k == "recon":
        return _recon_work(c["n"], c["n_gal"], c["n_gal"] * c["ratio"], 8 if c["dtype"] == "f64" else 4,
                           c["max_iter"] if c["tol"] == 0 else 12)
    if k == "batch":
        sides = [n for n in (32, 48, 64, 96, 128, 256, 384, 512) if c["n_lo"] <= n <= c["n_hi"]]
        g = (c["gal_lo"] + c["gal_hi"]) // 2
        ws = [_recon_work(sides[i % len(sides)], g, g * c["ratio"] if i % 2 == 0 else 0, 8, 12) for i in range(c["count"])]
        return {q: sum(w[q] for w in ws) for q in ("bytes", "flops")}
    if k == "shift":
        es = 8 if c["dtype"] == "f64" else 4
        return dict(bytes=c["count"] * (3 * es + 12 + 24) + 12.0 * min(c["n"] ** 3, 8 * c["count"]), flops=c["count"] * 100.0)
    if k == "frontend":
        es = 8 if c["dtype"] == "f64" else 4
        return dict(bytes=c["n_gal"] * (1 + c["ratio"]) * (3 * es + 4.0) + c["n"] ** 3 * 16.0,
                    flops=c["n_gal"] * (1 + c["ratio"]) * 30.0)
    if k == "fd":
        # about 8 iterations: two operator and two preconditioner applications each
        return dict(bytes=c["n"] ** 3 * 8.0 * 8 * 4, flops=8 * 2 * c["n"] ** 3 * (60.0 + 2 * 7.5 * math.log2(c["n"])))
    v, c1 = c["n"] ** 3, c["c1"]
    if k == "infer":
        return dict(bytes=v * 24.0, flops=_net_flops(c["n"], c1))
    # each activation written by the forward pass and read once by the backward pass
    acts = v * (4 * c1) + v // 8 * (8 * c1) + v // 64 * (8 * c1)
    return dict(bytes=v * 28.0 + acts * 2 * (2.0 if c["bf16"] else 4.0), flops=3 * _net_flops(c["n"], c1))


# ---- the same values in float64 -----------------------------------------------------------------
_CHUNK = 1 << 22


def _corners(pos, n, L):
    u = pos.double() * (n / L)
    i0 = torch.floor(u)
    t = u - i0
    i0 = i0.long()
    for dx in (0, 1):
        for dy in (0, 1):
            for dz in (0, 1):
                w = (t[:, 0] if dx else 1 - t[:, 0]) * (t[:, 1] if dy else 1 - t[:, 1]) * (t[:, 2] if dz else 1 - t[:, 2])
                yield (((i0[:, 0] + dx) % n) * n + (i0[:, 1] + dy) % n) * n + (i0[:, 2] + dz) % n, w


def _deposit64(pos, n, L):
    rho = torch.zeros(n ** 3, device="cuda", dtype=torch.float64)
    for p in pos.split(_CHUNK):
        for idx, w in _corners(p, n, L):
            rho.index_add_(0, idx, w)
    return rho.view(n, n, n)


def _waves(n, L):
    k1 = 2 * math.pi / L * torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64)
    kz = 2 * math.pi / L * torch.arange(n // 2 + 1, device="cuda", dtype=torch.float64)
    k = (k1[:, None, None], k1[None, :, None], kz[None, None, :])
    d1, dz = k1.clone(), kz.clone()
    d1[n // 2] = 0.0
    dz[n // 2] = 0.0
    return k, (d1[:, None, None], d1[None, :, None], dz[None, None, :])


def _delta64(p, gal, ran):
    """(delta, its transform) after smoothing, the mask and the logarithm."""
    n, L = p["n"], p["L"]
    k, _ = _waves(n, L)
    S = [torch.exp(-0.5 * a * a * p["R"] ** 2) for a in k]

    def smooth(rho):
        A = torch.fft.rfftn(rho)
        for s in S:
            A *= s
        return torch.fft.irfftn(A, s=(n, n, n))

    rg = smooth(_deposit64(gal, n, L))
    if p["uniform"]:
        q = rg * (n ** 3 / len(gal))
    else:
        rho_r = _deposit64(ran, n, L)
        touched = int((rho_r > 0).sum())
        rr = smooth(rho_r)
        mask = rr > p["mask_frac"] * len(ran) / touched
        q = torch.where(mask, rg * (len(ran) / len(gal)) / torch.where(mask, rr, 1.0), 1.0)
    d = q - 1
    if p["lognormal"]:
        d = torch.log(q.clamp_min(1e-6))
        d -= d.mean()
    return d


def _los64(p):
    """The three components of the line of sight, broadcastable, and 1/|d|."""
    n, L = p["n"], p["L"]
    o = torch.tensor(p["observer"], device="cuda", dtype=torch.float64)
    if p["los_mode"] == B.LOS_FIXED:
        return [v for v in o / torch.linalg.norm(o)], 1.0
    x = torch.arange(n, device="cuda", dtype=torch.float64) * (L / n)
    d = [(x - o[0])[:, None, None], (x - o[1])[None, :, None], (x - o[2])[None, None, :]]
    r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
    return d, torch.where(r2 > 0, r2.clamp_min(1e-300).rsqrt(), 0.0)


def _iterate64(p, d, start, tol, max_iter):
    n, L, beta = p["n"], p["L"], p["f"] / p["b"]
    k, kd = _waves(n, L)
    k2 = k[0] * k[0] + k[1] * k[1] + k[2] * k[2]
    k2[0, 0, 0] = 1.0
    inv = 1.0 / k2
    kd2 = (kd[0] * kd[0] + kd[1] * kd[1] + kd[2] * kd[2]) * inv * inv
    kd2[..., 1:n // 2] *= 2
    del k2
    Db = torch.fft.rfftn(d / p["b"])
    Db[0, 0, 0] = 0
    dv, w = _los64(p)
    back = lambda A: torch.fft.irfftn(A, s=(n, n, n))  # noqa: E731

    def source(S, coef):
        """delta/b + beta div(coef (Z[S].r) r)"""
        u = 0.0
        for j in range(3):
            u = u + back(S * (1j * kd[j]) * inv) * dv[j]
        u = u * w * w * coef
        out = Db.clone()
        for j in range(3):
            out += torch.fft.rfftn(u * dv[j]) * (1j * beta * kd[j])
        out[0, 0, 0] = 0
        return out

    c0 = {"plain": 0.0, "approx1": beta / (1 + beta)}.get(start, 3 * beta / (7 + 3 * beta))
    S, coef, it = Db, 1.0 - c0, 0
    while it < max_iter:
        new = source(S, coef)
        coef = 1.0
        it += 1
        if tol > 0:
            D = new - S
            d2 = float((kd2 * (D.real * D.real + D.imag * D.imag)).sum())
            s2 = float((kd2 * (new.real * new.real + new.imag * new.imag)).sum())
        S = new
        if tol > 0 and it >= 2 and math.sqrt(d2 / s2) < tol:
            break
    return torch.stack([back(S * (1j * kd[j]) * inv) for j in range(3)]), it


def _shift64(p, psi, pos, galaxy):
    n, L = p["n"], p["L"]
    flat = psi.reshape(3, -1)
    o = torch.tensor(p["observer"], device="cuda", dtype=torch.float64)
    out = []
    for q in pos.split(_CHUNK):
        v = torch.zeros((len(q), 3), device="cuda", dtype=torch.float64)
        for idx, w in _corners(q, n, L):
            v += flat[:, idx].T * w[:, None]
        if galaxy:
            if p["los_mode"] == B.LOS_FIXED:
                r = (o / torch.linalg.norm(o)).expand_as(v)
            else:
                x = torch.remainder(q.double(), L) - o
                r = x / torch.linalg.norm(x, dim=1, keepdim=True)
            v = v + p["f"] * (v * r).sum(1, keepdim=True) * r
        out.append(-v)
    return torch.cat(out)


def _fd64(p, d, tol):
    """BiCGStab in float64 on the operator of the finite-difference method, phi = 0 outside."""
    n, L, beta = p["n"], p["L"], p["f"] / p["b"]
    g = L / n
    dv, w = _los64(p)
    fixed = p["los_mode"] == B.LOS_FIXED
    iw2 = 1.0 if fixed else w * w

    def apply(phi):
        e = torch.nn.functional.pad(phi, (1, 1, 1, 1, 1, 1))
        at = lambda a, b, c: e[1 + a:n + 1 + a, 1 + b:n + 1 + b, 1 + c:n + 1 + c]  # noqa: E731
        unit = [(1, 0, 0), (0, 1, 0), (0, 0, 1)]
        face = [(at(*u), at(*(-v for v in u))) for u in unit]
        lap = (-6.0 * phi + sum(a + b for a, b in face)) / g ** 2
        rsd = -2.0 * phi / g ** 2 * (1.0 if fixed else (w > 0))
        for j in range(3):
            c2 = dv[j] * dv[j] * iw2 / g ** 2
            c1 = 0.0 if fixed else dv[j] * iw2 / g
            rsd = rsd + (c2 + c1) * face[j][0] + (c2 - c1) * face[j][1]
        for i in range(3):
            for j in range(i + 1, 3):
                cc = dv[i] * dv[j] * iw2 * 0.5 / g ** 2
                for si in (1, -1):
                    for sj in (1, -1):
                        o = [0, 0, 0]
                        o[i], o[j] = si, sj
                        rsd = rsd + si * sj * cc * at(*o)
        return lap + beta * rsd

    m = torch.arange(n, device="cuda", dtype=torch.float64)
    c1 = 2 * torch.cos(2 * math.pi * m / n) - 2
    lam = (c1[:, None, None] + c1[None, :, None] + c1[None, None, :n // 2 + 1]) / g ** 2
    lam[0, 0, 0] = -3 * math.pi ** 2 / L ** 2
    pre = lambda v: torch.fft.irfftn(torch.fft.rfftn(v) / lam, s=(n, n, n))  # noqa: E731
    b = d / p["b"]
    x, r = torch.zeros_like(b), b.clone()
    rh, q, bn = r.clone(), r.clone(), float(b.norm())
    rho = float((rh * r).sum())
    for _ in range(200):
        y = pre(q)
        v = apply(y)
        a = rho / float((rh * v).sum())
        s = r - a * v
        if float(s.norm()) / bn <= tol:
            x += a * y
            break
        z = pre(s)
        t = apply(z)
        om = float((t * s).sum()) / float((t * t).sum())
        x += a * y + om * z
        r = s - om * t
        if float(r.norm()) / bn <= tol:
            break
        new = float((rh * r).sum())
        q = r + new / rho * a / om * (q - om * v)
        rho = new
    e = torch.nn.functional.pad(x, (1, 1, 1, 1, 1, 1))
    h = 0.5 / g
    return torch.stack([-(e[2:, 1:-1, 1:-1] - e[:-2, 1:-1, 1:-1]) * h, -(e[1:-1, 2:, 1:-1] - e[1:-1, :-2, 1:-1]) * h,
                        -(e[1:-1, 1:-1, 2:] - e[1:-1, 1:-1, :-2]) * h])


def _net64(flat, specs, x, t):
    """(output, loss, gradients) of the network in float64, or the output alone without a target."""
    n = x.shape[0]
    prm = torch.from_numpy(flat).cuda().double()
    prm.requires_grad_(t is not None)
    layers, o = [], 0
    for ci, co, taps in specs:
        w = prm[o:o + taps * ci * co].view(taps, ci, co)
        o += taps * ci * co
        layers.append((w, prm[o:o + co]))
        o += co

    def conv(i, a, act=True):
        w, b = layers[i]
        if w.shape[0] == 1:
            return a @ w[0] + b
        y = b
        for s in range(27):
            off = (1 - s // 9, 1 - (s // 3) % 3, 1 - s % 3)
            y = y + torch.roll(a, off, (0, 1, 2)) @ w[s]
        return torch.relu(y) if act else y

    def pool(a):
        m = a.shape[0] // 2
        return a.view(m, 2, m, 2, m, 2, -1).mean((1, 3, 5))

    def up(a):
        return a.repeat_interleave(2, 0).repeat_interleave(2, 1).repeat_interleave(2, 2)

    xd = x.double()
    e1 = conv(1, conv(0, xd))
    e2 = conv(3, conv(2, pool(e1)))
    bt = conv(5, conv(4, pool(e2)))
    d2 = conv(7, conv(6, torch.cat([up(bt), e2], -1)))
    d1 = conv(9, conv(8, torch.cat([up(d2), e1], -1)))
    y = conv(10, d1)[..., 0] + xd[..., 4]
    if t is None:
        return y.view(n, n, n)
    loss = ((y - t.double()) ** 2).mean()
    loss.backward()
    return prm.detach(), float(loss.detach()), prm.grad


def exact(case, seed):
    c, k = case, case["kind"]
    if k == "recon":
        p, gal, ran = _mock(c, seed)
        psi, _ = _iterate64(p, _delta64(p, gal, None if p["uniform"] else ran), c["start"], c["tol"], c["max_iter"])
        out = dict(n_iter=None, shift_gal=_shift64(p, psi, gal, True))
        if ran is not None:
            out["shift_ran"] = _shift64(p, psi, ran, False)
        out["psi"] = psi
        return out
    if k == "batch":
        out = []
        for m in _batch_mocks(c, seed):
            p, gal, ran = m["params"], m["gal"], m["ran"]
            psi, _ = _iterate64(p, _delta64(p, gal, ran), "approx2", 1e-6, 80)
            out.append([None, _shift64(p, psi, gal, True), None if ran is None else _shift64(p, psi, ran, False)])
        return out
    if k == "shift":
        p, gal, pos = _shift_inputs(c, seed)
        psi, _ = _iterate64(p, _delta64(p, gal, None), "approx2", 0.0, 3)
        d = _shift64(p, psi, pos, c["galaxy"])
        y = pos.double() + d
        return dict(shift=d, pos=torch.remainder(y, c["L"]) if c["periodic"] else y)
    if k == "frontend":
        m = mocks.batch_mock_device(c["n"], c["n_gal"], c["ratio"], 1.85, 0.74, True, seed, L=c["L"])
        rmin, rmax, area = _shells(c)
        o = torch.tensor(m["params"]["observer"], device="cuda", dtype=torch.float64)
        nb, out, n = c["nbins"], {}, c["n"]

        def bins(pos):
            b = torch.floor((torch.linalg.norm(pos - o, dim=1) - rmin) * (nb / (rmax - rmin)))
            return torch.where((b >= 0) & (b < nb), b, float(nb)).long()

        gal, ran = _cast(m["gal"], c["dtype"]).double(), _cast(m["ran"], c["dtype"]).double()
        e = rmin + (rmax - rmin) / nb * torch.arange(nb + 1, device="cuda", dtype=torch.float64)
        nbar = torch.bincount(bins(gal), minlength=nb + 1)[:nb] / (area * (e[1:] ** 3 - e[:-1] ** 3) / 3)
        table = 1 / (1 + 20000.0 * torch.cat([nbar, nbar.new_zeros(1)]))
        for s, pos in (("gal", gal), ("ran", ran)):
            w = table[bins(pos)]
            i = torch.floor(pos * (n / c["L"]) + 0.5).long() % n
            out["w_" + s] = w
            out["rho_" + s] = torch.zeros(n ** 3, device="cuda", dtype=torch.float64).index_add_(
                0, (i[:, 0] * n + i[:, 1]) * n + i[:, 2], w).view(n, n, n)
        return dict(out, nbar=nbar)
    if k == "fd":
        p, gal = _fd_inputs(c, seed)
        return _fd64(p, _delta64(p, gal, None), 1e-9)
    flat, specs, x, t = _net_inputs(c, seed)
    if k == "infer":
        with torch.no_grad():
            return _net64(flat, specs, x, None)
    prm, loss, g = _net64(flat, specs, x, t)
    decay, o = torch.zeros_like(prm), 0
    for ci, co, taps in specs:
        decay[o:o + taps * ci * co] = 1.0
        o += taps * ci * co + co
    # the first AdamW step from zero moments
    new = prm - 1e-4 * (g / (g.abs() + 1e-8) + 1e-4 * decay * prm)
    return dict(loss=torch.tensor(loss, dtype=torch.float64), grads=g, params=new)
