"""The two-step kernels at the edges of their 4-column x 4-row items and of
their 64 x 64 tiles: padded sizes around multiples of 4 and 64, no sponge,
windows at every offset modulo 4, sources and receivers on tile borders.  The
one-step kernels compute the same operations, so records, gradients and images
agree bit for bit."""
import copy

import numpy as np
import pytest

import synth
from gpu_helpers import f32, f32_geom, gpu_ctx, to_dev, to_host

pytestmark = pytest.mark.gpu

# (nz, nx, nb): padded rows nz + 2 nb of 1, 4, 63 .. 66, 128, 131; windows of varied widths.
SHAPES = [(1, 9, 0), (4, 64, 0), (64, 65, 0), (23, 66, 20), (24, 67, 20), (25, 68, 20), (26, 129, 20), (88, 193, 20),
          (121, 203, 5), (150, 270, 64)]


def _case(nz, nx, nb):
    c = synth.tiny_case(nz=nz, nx=nx, nt=61, nb=nb, n_shots=1, seed=3)
    v = f32(1800.0 + 400.0 * synth.rng(7).uniform(size=(nz, nx)))
    g = copy.deepcopy(c.geom)
    # Window starts 0..3 modulo 4, widths that differ, record lengths odd and even.
    starts = [min(s, nx - 1) for s in (0, 1, 2, 3)]
    ends = [nx, nx, max(nx - 5, starts[2] + 1), max(nx - 2, starts[3] + 1)]
    zs = [z for z in (0, 43, 44, 63 - nb, 64 - nb) if 0 <= z < nz] or [0]
    rz, rx, off = [], [], [0]
    for s, (a, b) in enumerate(zip(starts, ends)):
        x = np.arange(a, b, 3)
        rx += list(x) + [a]  # two receivers share a cell
        rz += [zs[(s + i) % len(zs)] for i in range(len(x))] + [zs[s % len(zs)]]
        off.append(len(rx))
    i32 = lambda a: np.asarray(a, dtype=np.int32)
    g.src_iz = i32([zs[s % len(zs)] for s in range(4)])
    g.src_ix = i32([min(b - 1, max(a, min(64 - nb + a, b - 1)) if s % 2 else a) for s, (a, b) in
                    enumerate(zip(starts, ends))])
    g.nt = i32([61, 60, 59, 2])
    g.rec_off, g.rec_iz, g.rec_ix = i32(off), i32(rz), i32(rx)
    g.win_x0, g.win_x1 = i32(starts), i32(ends)
    c.geom = g
    return c, v


def _run(c, v, blocking, history, monkeypatch):
    import torch

    monkeypatch.setenv("DHFWI_STEP_VARIANT", "4")
    monkeypatch.setenv("DHFWI_TIME_BLOCK", "1" if blocking else "0")
    monkeypatch.setenv("DHFWI_HISTORY_MB", history) if history else monkeypatch.delenv("DHFWI_HISTORY_MB", raising=False)
    ctx = gpu_ctx(c)
    geom = f32_geom(c.geom)
    vd = to_dev(v)
    d = ctx.model_shots(vd, geom)
    ds = torch.empty(geom.n_data, dtype=torch.float32, device="cuda")
    J, g = ctx.fwi_gradient(vd, geom, 0.5 * d, d_syn=ds)
    b = ctx.born_demig(vd, geom, to_dev(f32(synth.gaussian_field(v.shape, seed=12))))
    m = ctx.rtm_mig(vd, geom, d)
    # Born from the forward pass that the gradient stored (all of it, or recomputed segments).
    ctx.set_reuse(True)
    ctx.fwi_gradient(vd, geom, 0.5 * d)
    br = ctx.born_demig(vd, geom, to_dev(f32(synth.gaussian_field(v.shape, seed=12))))
    assert ctx.stats()["reused"] == (0 if history else 2)
    out = [to_host(x) for x in (d, ds, g, b, m, br)] + [J]
    ctx.close()
    np.testing.assert_array_equal(out[3], out[5])
    return out


@pytest.mark.parametrize("history", ["", "0"], ids=["history", "recompute"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_two_steps_equal_one_step_at_the_edges(shape, history, monkeypatch):
    c, v = _case(*shape)
    one = _run(c, v, False, history, monkeypatch)
    two = _run(c, v, True, history, monkeypatch)
    assert np.all(np.isfinite(one[0])) and np.linalg.norm(one[0]) > 0 and np.linalg.norm(one[3]) > 0
    for a, b in zip(one, two):
        np.testing.assert_array_equal(a, b)
