"""A model of more than 2^31 padded cells with narrow windows: the two-step
kernels read kappa and its perturbation at rows past the 32-bit offsets, and agree
bit for bit with the one-step kernels, whose tensor maps address them."""
import types

import numpy as np
import pytest

from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu

NZ, NX, NB = 3250, 700000, 5  # padded 3260 rows of pitch 700032: rows from 3068 on start past 2^31
Z, X = 3130, NX - 100         # the part that the waves cross


def _geom():
    i32 = lambda a: np.asarray(a, dtype=np.int32)
    x0 = [X + 1, X + 30]
    rx = [np.arange(a, a + 60, 2) for a in x0]
    rz = [Z + 40 + (r % 60) for r in rx]
    t = (np.arange(41) - 12) * 0.15
    return types.SimpleNamespace(
        src_iz=i32([Z + 45, Z + 70]), src_ix=i32([X + 20, X + 61]), nt=i32([41, 40]), rec_off=i32([0, 30, 60]),
        rec_iz=i32(np.concatenate(rz)), rec_ix=i32(np.concatenate(rx)), win_x0=i32(x0), win_x1=i32([x0[0] + 61, NX]),
        wavelet=((1.0 - 2.0 * t * t) * np.exp(-t * t)).astype(np.float32), wavelet_shared=True)


def test_rows_past_32_bit_offsets(monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.mem_get_info()[0] < 140e9:
        pytest.skip("needs 140 GB of device memory")
    from paper_2403_17518_gb300 import build
    from paper_2403_17518_gb300.ops import Context

    build()
    monkeypatch.setenv("DHFWI_STEP_VARIANT", "4")
    rng = np.random.Generator(np.random.PCG64(5))
    part = rng.uniform(size=(2, NZ - Z, NX - X))
    v = torch.full((NZ, NX), 2000.0, device="cuda")
    v[Z:, X:] = to_dev(1800.0 + 400.0 * part[0])
    dv = torch.zeros((NZ, NX), device="cuda")
    dv[Z:, X:] = to_dev(50.0 * (part[1] - 0.5))
    g = _geom()
    ctx = Context(NZ, NX, 10.0, 1e-3, NB)
    out = {}
    for block in ("0", "1"):
        monkeypatch.setenv("DHFWI_TIME_BLOCK", block)
        d = ctx.model_shots(v, g)
        b = ctx.born_demig(v, g, dv)
        J, grad = ctx.fwi_gradient(v, g, 0.5 * d)
        out[block] = [d.cpu(), b.cpu(), grad[Z:, X:].cpu(), J]
        del grad
    ctx.close()
    del v, dv
    torch.cuda.empty_cache()
    one, two = out["0"], out["1"]
    for a, b in zip(one[:3], two[:3]):
        assert torch.isfinite(a).all() and a.abs().max() > 0
        assert torch.equal(a, b)
    assert one[3] == two[3]
