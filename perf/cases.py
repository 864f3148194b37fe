"""The framework's work as a user's program has it do: wave-equation operators on shot
gathers (forward modelling, gradient, Born demigration, migration, the operators of one
deblurred iteration) and the deblurring network (one training step, one full-image apply).

A case's geometry (sources, receivers, windows, record lengths) follows from the case alone;
models, data, network weights and images follow from the seed.
"""
import math
import types

import numpy as np
import torch

from paper_2403_17518_gb300.ops import Context, GeomArgs

NB = 20  # sponge cells
STENCIL = (-205.0 / 72.0, 8.0 / 5.0, -1.0 / 5.0, 8.0 / 315.0, -1.0 / 560.0)


def _wave(name, kind, nz, nx, h, dt, shots, nt, nt_min, nrec, nrec_min, f0, rec_step=1, margin=100, rel=False):
    """margin < 0: every shot sees the whole model width and every rec_step-th node of it; else
    nrec_min..nrec consecutive receivers about the source, window = their span and source +- margin."""
    return {"name": name, "kind": kind, "nz": nz, "nx": nx, "h": h, "dt": dt, "shots": shots, "nt": nt,
            "nt_min": nt_min, "nrec": nrec, "nrec_min": nrec_min, "rec_step": rec_step, "margin": margin,
            "f0": f0, "rel": rel}


def _net(name, kind, base, levels, n, h, w):
    return {"name": name, "kind": kind, "base": base, "levels": levels, "n": n, "h": h, "w": w}


def listed():
    return [
        # A quick look at a small two-layer-sized model: the smallest call, where launches count.
        _wave("model-101x101", "model", 101, 101, 10.0, 1e-3, 4, 500, 500, 51, 51, 15.0, rec_step=2, margin=-1),
        # One trial of a line search on the batched workload: every shot modelled, nothing stored.
        _wave("model-400x1200", "model", 400, 1200, 12.5, 1e-3, 64, 4000, 3000, 600, 200, 8.0),
        # The gradient of the small model: launches again, in both directions of time.
        _wave("gradient-101x101", "gradient", 101, 101, 10.0, 1e-3, 4, 500, 500, 51, 51, 15.0, rec_step=2, margin=-1),
        # The gradient at the Marmousi test's shape: fixed spread, full-width windows.
        _wave("gradient-221x601", "gradient", 221, 601, 15.0, 1.5e-3, 30, 2400, 2400, 300, 300, 5.0, rec_step=2,
              margin=-1),
        # A quarter of the batched workload's gradient: uneven windows, apertures and records.
        _wave("gradient-400x1200", "gradient", 400, 1200, 12.5, 1e-3, 16, 4000, 3000, 600, 200, 8.0),
        # Born demigration of an update direction over half of the batched workload.
        _wave("born-400x1200", "born", 400, 1200, 12.5, 1e-3, 32, 4000, 3000, 600, 200, 8.0),
        # Migration in the relative parameterisation at the FWI driver's default model.
        _wave("migrate-150x500", "migrate", 150, 500, 20.0, 2e-3, 25, 1500, 1200, 250, 166, 8.0, margin=50, rel=True),
        # The driver's operators of one deblurred iteration, the forward wavefield kept between them.
        _wave("iteration-150x500", "iteration", 150, 500, 20.0, 2e-3, 25, 1500, 1200, 250, 166, 8.0, margin=50),
        # One training step of the workload's network: a batch of 128 x 128 patches.
        _net("train-step-32x128x128", "net_grad", 32, 4, 32, 128, 128),
        # One full-image training step of the network at the paper's width.
        _net("train-step-base128", "net_grad", 128, 4, 1, 224, 608),
        # The update direction from a gradient of the batched workload's model.
        _net("apply-400x1200", "net_apply", 32, 4, 1, 400, 1200),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["model", "model", "gradient", "gradient", "born", "migrate", "iteration", "net_grad",
                       "net_apply"])
    if kind.startswith("net"):
        base = rng.choice([16, 32, 32, 64, 128])
        if kind == "net_apply":
            c = _net("", kind, base, 4, 1, log_int(96, 416), log_int(160, 1216))
        else:
            side = 16 * rng.randint(3, 10)
            most = max(1, 32 * 128 * 128 * 32 // (side * side * base))
            c = _net("", kind, base, 4, log_int(1, most), side, side if rng.random() < 0.5 else 16 * rng.randint(3, 10))
            if c["n"] * c["h"] * c["w"] * base > 32 * 128 * 128 * 32:
                c["n"] = max(1, 32 * 128 * 128 * 32 // (c["h"] * c["w"] * base))
    else:
        h = rng.choice([10.0, 12.5, 15.0, 20.0])
        dt = round(rng.uniform(0.3, 0.48) * h / 4700.0, 5)
        nz, nx = log_int(60, 420), log_int(90, 1220)
        shots, nt = log_int(2, 64), log_int(200, 4000)
        full = rng.random() < 0.4
        while True:
            nrec = max(20, int(nx * rng.uniform(0.25, 0.5)))
            c = _wave("", kind, nz, nx, h, dt, shots, nt, int(nt * rng.uniform(0.7, 1.0)), nrec,
                      max(10, int(nrec * rng.uniform(0.4, 1.0))), rng.choice([5.0, 8.0, 12.0]),
                      rec_step=rng.choice([1, 2]) if full else 1, margin=-1 if full else min(100, max(10, nx // 10)),
                      rel=kind in ("born", "migrate") and rng.random() < 0.5)
            # No more than the largest listed case; the stored history fits the card three times over.
            if _updates(c) <= 3.5e10 and (kind in ("model", "born") or _padded(c) <= 1.5e10):
                break
            shots, nt = max(1, shots * 3 // 4), max(150, nt * 7 // 8)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# Geometry and work
# ---------------------------------------------------------------------------
def _geometry(c):
    g = np.random.Generator(np.random.PCG64(17))
    nx, ns = c["nx"], c["shots"]
    edge = min(20, nx // 8)
    sx = np.rint(np.linspace(edge, nx - 1 - edge, ns)).astype(np.int64)
    nt = g.integers(c["nt_min"], c["nt"] + 1, ns)
    nt[0] = c["nt"]
    rec, x0, x1 = [], [], []
    for s in range(ns):
        if c["margin"] < 0:
            rec.append(np.arange(0, nx, c["rec_step"]))
            x0.append(0)
            x1.append(nx)
        else:
            n = min(nx, int(g.integers(c["nrec_min"], c["nrec"] + 1)))
            lo = max(0, min(int(sx[s]) - n // 2, nx - n))
            rec.append(np.arange(lo, lo + n))
            x0.append(max(0, min(lo, int(sx[s]) - c["margin"])))
            x1.append(min(nx, max(lo + n, int(sx[s]) + c["margin"] + 1)))
    rec_ix = np.concatenate(rec)
    t = np.arange(c["nt"]) * c["dt"] - 1.5 / c["f0"]
    a = (math.pi * c["f0"] * t) ** 2
    return types.SimpleNamespace(
        src_iz=np.zeros(ns, np.int32), src_ix=sx.astype(np.int32), nt=nt.astype(np.int32),
        rec_off=np.concatenate([[0], np.cumsum([len(r) for r in rec])]).astype(np.int32),
        rec_iz=np.zeros(len(rec_ix), np.int32), rec_ix=rec_ix.astype(np.int32),
        win_x0=np.asarray(x0, np.int32), win_x1=np.asarray(x1, np.int32),
        wavelet=((1.0 - 2.0 * a) * np.exp(-a)).astype(np.float32), wavelet_shared=True)


def _sweeps(kind):
    """Cell updates of a pass in units of one forward modelling of its shots."""
    return {"model": 1, "gradient": 2, "born": 2, "migrate": 2, "iteration": 4}[kind]


def _updates(c):
    g = _geometry(c)
    w = (g.win_x1 - g.win_x0).astype(np.int64) + 2 * NB
    return _sweeps(c["kind"]) * int(np.sum(g.nt.astype(np.int64) * (c["nz"] + 2 * NB) * w))


def _padded(c):
    g = _geometry(c)
    w = int((g.win_x1 - g.win_x0).max()) + 2 * NB + 63
    return int(g.nt.astype(np.int64).sum()) * (c["nz"] + 2 * NB) * w


def _net_layers(base, levels):
    """(kind, input channels, output channels, level the layer's input lives on)."""
    c = [base << r for r in range(levels + 1)]
    out = [("c3", 1, c[0], 0), ("c3", c[0], c[0], 0)]
    for r in range(1, levels + 1):
        out += [("c3", c[r - 1], c[r], r), ("c3", c[r], c[r], r)]
    for r in range(levels - 1, -1, -1):
        out += [("ct", c[r + 1], c[r], r + 1), ("c3", 2 * c[r], c[r], r), ("c3", c[r], c[r], r)]
    return out + [("c1", c[0], 1, 0)]


TAPS = {"c3": 9, "ct": 4, "c1": 1}


def work(case):
    """Inputs read once and outputs written once.  A cell update of the recurrence takes 26 operations
    (20 for the four neighbour rings, 1 for the centre, 5 for the damped update); a network layer two per
    multiply-add, three times over for a training step (output, input and weight gradients)."""
    kind = case["kind"]
    if kind.startswith("net"):
        layers = _net_layers(case["base"], case["levels"])
        m = 1 << case["levels"]
        h, w = -(-case["h"] // m) * m, -(-case["w"] // m) * m
        flops = sum(2.0 * case["n"] * (h >> r) * (w >> r) * TAPS[k] * ci * co for k, ci, co, r in layers)
        params = sum(TAPS[k] * ci * co + co for k, ci, co, _ in layers)
        pixels = case["n"] * case["h"] * case["w"]
        if kind == "net_grad":
            return {"bytes": 4.0 * (2 * pixels + 2 * params), "flops": 3.0 * flops}
        return {"bytes": 4.0 * (2 * pixels + params), "flops": flops}
    g = _geometry(case)
    model = case["nz"] * case["nx"]
    data = int(np.sum(g.nt.astype(np.int64) * np.diff(g.rec_off)))
    values = {"model": model + data, "gradient": 2 * model + 2 * data, "born": 2 * model + data,
              "migrate": 2 * model + data, "iteration": 3 * model + 3 * data}[kind]
    return {"bytes": 4.0 * values, "flops": 26.0 * _updates(case)}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _gen(seed, salt):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 16 + salt)


def _blur(f, sigma):
    """Gaussian smoothing along both axes, edges repeated."""
    r = int(3 * sigma)
    k = [math.exp(-0.5 * (t / sigma) ** 2) for t in range(-r, r + 1)]
    for axis in (0, 1):
        n = f.shape[axis]
        at = torch.arange(n, device=f.device)
        f = sum(f.index_select(axis, (at + t).clamp(0, n - 1)) * (c / sum(k)) for t, c in zip(range(-r, r + 1), k))
    return f.contiguous()


def _model(case, seed):
    """Layers of 1500 to 4500 m/s with dips and a smooth perturbation, smoothed as an initial model is."""
    g = _gen(seed, 0)
    nz, nx = case["nz"], case["nx"]
    dev = torch.device("cuda")
    z = torch.arange(nz, device=dev, dtype=torch.float32)[:, None] / nz
    x = torch.arange(nx, device=dev, dtype=torch.float32)[None, :] / nx
    r = torch.rand(3, 8, device=dev, generator=g)
    tops = torch.sort(0.05 + 0.9 * r[0]).values
    depth = (z[None] > tops[:, None, None] + 0.2 * (r[1] - 0.5)[:, None, None] * (x - r[2][:, None, None]))
    v = 1500.0 + 375.0 * depth.sum(0).float()
    v = v + 100.0 * torch.randn(nz, nx, device=dev, generator=g)
    return _blur(v, 4.0).clamp(1500.0, 4500.0).contiguous()


def _field(case, seed, amplitude):
    f = _blur(torch.randn(case["nz"], case["nx"], device="cuda", generator=_gen(seed, 1)), 3.0)
    return (f * (amplitude / f.abs().max())).contiguous()


def _records(case, geom, seed, scale=1.0):
    """A direct wave and eight reflections per trace, with the moveout and the decay with distance of
    point-source records, and a little noise."""
    gen = _gen(seed, 2)
    dev = torch.device("cuda")
    r = torch.rand(3, 9, device=dev, generator=gen).cpu().numpy()
    out, off = [], geom.rec_off
    for s in range(len(geom.nt)):
        nt = int(geom.nt[s])
        x = np.abs(geom.rec_ix[off[s]:off[s + 1]].astype(np.float64) - float(geom.src_ix[s])) * case["h"]
        x = torch.as_tensor(x, device=dev, dtype=torch.float32)[None, :]
        t = (torch.arange(nt, device=dev, dtype=torch.float32)[:, None] + 1.0) * case["dt"] - 1.5 / case["f0"]
        d = torch.zeros(nt, x.shape[1], device=dev)
        for k in range(9):
            t0 = 0.0 if k == 0 else (0.1 + 0.85 * r[0, k]) * nt * case["dt"]
            vel = 1500.0 if k == 0 else 1600.0 + 2000.0 * r[1, k]
            amp = 1.0 if k == 0 else 0.2 * (r[2, k] - 0.5)
            ta = torch.sqrt(t0 * t0 + (x / vel) ** 2)
            a = (math.pi * case["f0"] * (t - ta)) ** 2
            d += amp * 0.02 * torch.rsqrt((vel * ta + 2.0 * case["h"]) / 1000.0) * (1.0 - 2.0 * a) * torch.exp(-a)
        out.append(d.reshape(-1))
    d = torch.cat(out)
    d += 2e-5 * torch.randn(d.shape, device=dev, generator=gen)
    return (d * scale).contiguous()


def _weights(case, seed):
    """Kaiming-uniform weights and biases in the flat parameter layout."""
    g = _gen(seed, 3)
    parts = []
    for k, ci, co, _ in _net_layers(case["base"], case["levels"]):
        bound = 1.0 / math.sqrt(ci * (9 if k == "c3" else 1))
        parts.append((torch.rand(TAPS[k] * ci * co + co, device="cuda", generator=g) * 2.0 - 1.0) * bound)
    return torch.cat(parts)


def _images(case, seed, salt):
    """Smooth images of unit size, as normalised gradients and migrated images are."""
    x = torch.randn(case["n"], 1, case["h"], case["w"], device="cuda", generator=_gen(seed, salt))
    x = torch.nn.functional.avg_pool2d(x, 5, stride=1, padding=2)
    return (x[:, 0] / x.abs().amax()).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    st = types.SimpleNamespace(kind=kind)
    if kind.startswith("net"):
        st.ctx = Context(case["h"], case["w"], 10.0, 1e-3, NB)
        st.ctx.net_init(case["base"], case["levels"], 29)
        st.ctx.net_set(_weights(case, seed).cpu().numpy())
        st.x = _images(case, seed, 4)
        if kind == "net_grad":
            st.y = _images(case, seed, 5)
        else:
            st.x = st.x[0].contiguous()
            st.out = torch.empty_like(st.x)
        return st
    geom = _geometry(case)
    st.ctx = Context(case["nz"], case["nx"], case["h"], case["dt"], NB)
    st.geom = GeomArgs(geom)
    st.rel = case["rel"]
    st.v = _model(case, seed)
    if kind in ("model", "born"):
        st.data = st.ctx.new_data(st.geom)
    else:
        st.data = _records(case, geom, seed, 1e-2 if kind == "migrate" else 1.0)
        st.img = st.ctx.new_model()
    if kind == "born":
        st.dv = _field(case, seed, 0.05 if st.rel else 150.0)
    if kind == "iteration":
        st.ctx.set_reuse(True)
        st.born = st.ctx.new_data(st.geom)
        st.dm = st.ctx.new_model()
    return st


def run(st):
    c = st.ctx
    if st.kind == "model":
        return [c.model_shots(st.v, st.geom, out=st.data)]
    if st.kind == "gradient":
        misfit, grad = c.fwi_gradient(st.v, st.geom, st.data, grad=st.img)
        return [np.float32(misfit), grad]  # a sum over float32 records: as exact as they are
    if st.kind == "born":
        return [c.born_demig(st.v, st.geom, st.dv, rel=st.rel, out=st.data)]
    if st.kind == "migrate":
        return [c.rtm_mig(st.v, st.geom, st.data, rel=st.rel, out=st.img)]
    if st.kind == "iteration":
        misfit, grad = c.fwi_gradient(st.v, st.geom, st.data, grad=st.img)
        born = c.born_demig(st.v, st.geom, grad, out=st.born)
        return [np.float32(misfit), grad, born, c.rtm_mig(st.v, st.geom, born, out=st.dm)]
    if st.kind == "net_grad":
        loss, grad = c.deblur_grad(st.x, st.y)
        return [np.float32(loss), grad]
    return [c.deblur_apply(st.x, out=st.out)]


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------
class _Exact:
    """The recurrence of the propagators in float64, all shots of a case at once."""

    def __init__(self, case, v):
        g = self.g = _geometry(case)
        dev = self.dev = v.device
        ns, NZ = len(g.nt), case["nz"] + 2 * NB
        width = (g.win_x1 - g.win_x0 + 2 * NB).astype(np.int64)
        W = int(width.max())
        self.shape = (ns, NZ, W)
        self.nt = int(g.nt.max())
        rows = np.clip(np.arange(NZ) - NB, 0, case["nz"] - 1)
        cols = np.clip(g.win_x0[:, None].astype(np.int64) + np.arange(W)[None, :] - NB, 0, case["nx"] - 1)
        self.cell = torch.as_tensor(rows[None, :, None] * case["nx"] + cols[:, None, :], device=dev)
        self.v = v.double()
        c = float(np.float32(case["dt"])) ** 2 / float(np.float32(case["h"])) ** 2
        self.kappa = (c * self.v * self.v).reshape(-1)[self.cell]

        def sponge(n, size):
            d = np.minimum(np.arange(size), n - 1 - np.arange(size))
            f = np.exp(-(0.015 * np.maximum(NB - d, 0)) ** 2)
            return np.where((np.arange(size) < n), f, 0.0)  # zero outside the window

        wx = np.stack([sponge(int(n), W) for n in width])
        self.w = torch.as_tensor(sponge(NZ, NZ)[None, :, None] * wx[:, None, :], device=dev)
        sh = np.repeat(np.arange(ns), np.diff(g.rec_off))
        self.rec = (torch.as_tensor(sh, device=dev), torch.as_tensor(g.rec_iz.astype(np.int64) + NB, device=dev),
                    torch.as_tensor(g.rec_ix.astype(np.int64) - g.win_x0[sh] + NB, device=dev))
        self.src = (torch.arange(ns, device=dev), torch.as_tensor(g.src_iz.astype(np.int64) + NB, device=dev),
                    torch.as_tensor(g.src_ix.astype(np.int64) - g.win_x0 + NB, device=dev))
        self.wav = torch.as_tensor(g.wavelet.astype(np.float64), device=dev)

    def state(self):
        ns, NZ, W = self.shape
        u = torch.zeros(ns, NZ + 8, W + 8, dtype=torch.float64, device=self.dev)
        return u, torch.zeros(self.shape, dtype=torch.float64, device=self.dev)

    def lap(self, u, out):
        NZ, W = self.shape[1:]
        torch.mul(u[:, 4:4 + NZ, 4:4 + W], 2.0 * STENCIL[0], out=out)
        for k in range(1, 5):
            for s in (u[:, 4 - k:4 - k + NZ, 4:4 + W], u[:, 4 + k:4 + k + NZ, 4:4 + W],
                      u[:, 4:4 + NZ, 4 - k:4 - k + W], u[:, 4:4 + NZ, 4 + k:4 + k + W]):
                out.add_(s, alpha=STENCIL[k])
        return out

    def advance(self, u, d):
        NZ, W = self.shape[1:]
        d.mul_(self.w)
        uc = u[:, 4:4 + NZ, 4:4 + W]
        uc.mul_(self.w).add_(d)
        return uc

    def pack(self, samples):
        """[nt][all receivers] to the packed layout, shot after shot."""
        off = self.g.rec_off
        return torch.cat([samples[:int(self.g.nt[s]), off[s]:off[s + 1]].reshape(-1) for s in range(len(self.g.nt))])

    def unpack(self, d):
        off, at = self.g.rec_off, 0
        out = torch.zeros(self.nt, int(off[-1]), dtype=torch.float64, device=self.dev)
        for s in range(len(self.g.nt)):
            n, m = int(self.g.nt[s]), int(off[s + 1] - off[s])
            out[:n, off[s]:off[s + 1]] = d[at:at + n * m].double().view(n, m)
            at += n * m
        return out

    def forward(self, keep):
        u, d = self.state()
        a = torch.empty(self.shape, dtype=torch.float64, device=self.dev)
        hist = torch.empty((self.nt,) + self.shape, dtype=torch.float64, device=self.dev) if keep else None
        out = torch.zeros(self.nt, len(self.rec[0]), dtype=torch.float64, device=self.dev)
        for n in range(self.nt):
            a = self.lap(u, hist[n] if keep else a)
            a[self.src] += self.wav[n]
            d.addcmul_(self.kappa, a)
            out[n] = self.advance(u, d)[self.rec]
        return self.pack(out), hist

    def born(self, dkappa):
        u, d = self.state()
        p, dp = self.state()
        a = torch.empty(self.shape, dtype=torch.float64, device=self.dev)
        b = torch.empty_like(a)
        out = torch.zeros(self.nt, len(self.rec[0]), dtype=torch.float64, device=self.dev)
        for n in range(self.nt):
            self.lap(u, a)
            a[self.src] += self.wav[n]
            dp.addcmul_(self.kappa, self.lap(p, b)).addcmul_(dkappa, a)
            d.addcmul_(self.kappa, a)
            self.advance(u, d)
            out[n] = self.advance(p, dp)[self.rec]
        return self.pack(out)

    def dkappa(self, dv, rel):
        return 2.0 * self.kappa * (dv.double() if rel else dv.double() / self.v).reshape(-1)[self.cell]

    def image(self, hist, data, rel):
        nu, d = self.state()
        a = torch.empty(self.shape, dtype=torch.float64, device=self.dev)
        img = torch.zeros(self.shape, dtype=torch.float64, device=self.dev)
        r = self.unpack(data)
        for k in range(self.nt, 0, -1):
            self.lap(nu, a)
            a.index_put_(self.rec, r[k - 1], accumulate=True)
            d.addcmul_(self.kappa, a)
            img.addcmul_(hist[k - 1], self.advance(nu, d))
        out = torch.zeros(self.v.numel(), dtype=torch.float64, device=self.dev)
        out.index_add_(0, self.cell.reshape(-1), img.reshape(-1))
        return out.view_as(self.v) * (2.0 if rel else 2.0 / self.v)


def _exact_net(case, theta, x):
    """The U-Net in float64: the output and the leaf parameters it was computed from."""
    F = torch.nn.functional
    leaves, at = [], 0
    for k, ci, co, _ in _net_layers(case["base"], case["levels"]):
        n = TAPS[k] * ci * co
        w = theta[at:at + n].double().requires_grad_()
        b = theta[at + n:at + n + co].double().requires_grad_()
        leaves.append((k, ci, co, w, b))
        at += n + co
    it = iter(leaves)

    def layer(h):
        k, ci, co, w, b = next(it)
        if k == "ct":  # weight [co][2][2][ci]
            return F.conv_transpose2d(h, w.view(co, 2, 2, ci).permute(3, 0, 1, 2), b, stride=2)
        if k == "c1":
            return F.conv2d(h, w.view(co, ci, 1, 1), b)
        return F.leaky_relu(F.conv2d(h, w.view(co, 3, 3, ci).permute(0, 3, 1, 2), b, padding=1), 0.2)

    h, skips = layer(layer(x.double()[:, None])), []
    for _ in range(case["levels"]):
        skips.append(h)
        h = layer(layer(F.avg_pool2d(h, 3, stride=2, padding=1)))
    for _ in range(case["levels"]):
        h = layer(torch.cat([skips.pop(), layer(h)], 1))
        h = layer(h)
    return layer(h)[:, 0], [t for _, _, _, w, b in leaves for t in (w, b)]


def exact(case, seed):
    kind = case["kind"]
    if kind.startswith("net"):
        theta = _weights(case, seed)
        x = _images(case, seed, 4)
        if kind == "net_grad":
            out, leaves = _exact_net(case, theta, x)
            loss = torch.mean((out - _images(case, seed, 5).double()) ** 2)
            grads = torch.autograd.grad(loss, leaves)
            return [loss.detach(), torch.cat([g.reshape(-1) for g in grads])]
        m = 1 << case["levels"]
        scale = x.abs().max().double()
        pad = (0, -case["w"] % m, 0, -case["h"] % m)
        with torch.no_grad():
            out, _ = _exact_net(case, theta, torch.nn.functional.pad(x.double() / scale, pad))
        return [(out[0, :case["h"], :case["w"]] * scale).contiguous()]
    with torch.no_grad():
        v = _model(case, seed)
        e = _Exact(case, v)
        if kind == "model":
            return [e.forward(False)[0]]
        if kind == "born":
            return [e.born(e.dkappa(_field(case, seed, 0.05 if case["rel"] else 150.0), case["rel"]))]
        d_obs = _records(case, e.g, seed, 1e-2 if kind == "migrate" else 1.0)
        d_syn, hist = e.forward(True)
        if kind == "migrate":
            return [e.image(hist, d_obs, case["rel"])]
        r = d_syn - d_obs.double()
        misfit, grad = 0.5 * (r * r).sum(), e.image(hist, r, False)
        if kind == "gradient":
            return [misfit, grad]
        born = e.born(e.dkappa(grad, False))
        return [misfit, grad, born, e.image(hist, born, False)]
