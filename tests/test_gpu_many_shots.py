"""More shots than a grid's second dimension takes (65535): every call runs, every
shot's record is one shot's, and one and two steps per launch agree bit for bit."""
import types

import numpy as np
import pytest

import synth
from gpu_helpers import f32, gpu_ctx, to_dev, to_host

pytestmark = pytest.mark.gpu

N = 65600


def _geom(k):
    i32 = lambda a: np.asarray(a, dtype=np.int32)
    return types.SimpleNamespace(
        src_iz=i32([1] * k), src_ix=i32([4] * k), nt=i32([5] * k), rec_off=i32(range(0, 2 * k + 1, 2)),
        rec_iz=i32([0, 2] * k), rec_ix=i32([2, 7] * k), win_x0=i32([0] * k), win_x1=i32([9] * k),
        wavelet=np.array([1.0, -2.0, 0.5, 0.0, 1.0], dtype=np.float32), wavelet_shared=True)


def test_more_shots_than_a_grid_dimension(monkeypatch):
    c = synth.tiny_case(nz=3, nx=9, nt=5, nb=1, n_shots=1, seed=3)
    v = to_dev(f32(1800.0 + 400.0 * synth.rng(7).uniform(size=(3, 9))))
    one, many = _geom(1), _geom(N)
    grads = []
    for block in ("0", "1"):
        monkeypatch.setenv("DHFWI_TIME_BLOCK", block)
        ctx = gpu_ctx(c)
        d1 = ctx.model_shots(v, one)
        b1 = to_host(ctx.born_demig(v, one, 0.01 * v))
        J1, _ = ctx.fwi_gradient(v, one, 0.5 * d1)
        d = ctx.model_shots(v, many)
        b = to_host(ctx.born_demig(v, many, 0.01 * v))
        J, g = ctx.fwi_gradient(v, many, 0.5 * d)
        ctx.close()
        grads.append(to_host(g))
        d1 = to_host(d1)
        assert np.linalg.norm(d1) > 0 and np.linalg.norm(b1) > 0 and np.linalg.norm(grads[-1]) > 0
        np.testing.assert_array_equal(to_host(d).reshape(N, -1), np.broadcast_to(d1, (N, d1.size)))
        np.testing.assert_array_equal(b.reshape(N, -1), np.broadcast_to(b1, (N, b1.size)))
        assert abs(J - N * J1) <= 1e-9 * J  # float64 sums of 656 000 equal-sized terms
    np.testing.assert_array_equal(grads[0], grads[1])
