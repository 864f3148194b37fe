"""Two-step launches of many step pairs: plans with more tiles than resident CTAs,
so that tiles wait for their neighbours' progress inside a launch.  Records of
uneven, odd and even lengths join and leave in mid-launch, and the longest takes a
full launch of 256 pairs and a short one, of twelve pairs or of one.  The one-step
kernels compute the same operations, so records, gradients and images agree bit for
bit."""
import copy

import numpy as np
import pytest

import synth
from gpu_helpers import f32, f32_geom, gpu_ctx, to_dev
from test_gpu_pair_edges import _run

pytestmark = pytest.mark.gpu

# The longest record: 512 steps, then 23 or 1 (a launch of one pair after one of many).
NT = {56: 535, 130: 513}


def _case(n_shots):
    """Windows of 2 x 3 or 3 x 3 tiles (padded rows 160), four of them of every
    offset modulo 4; half of the records nearly as long as the longest."""
    nz, nx, nb = 150, 181, 5
    nt = NT[n_shots]
    c = synth.tiny_case(nz=nz, nx=nx, nt=nt, nb=nb, n_shots=1, seed=3)
    v = f32(1800.0 + 400.0 * synth.rng(7).uniform(size=(nz, nx)))
    g = copy.deepcopy(c.geom)
    i32 = lambda a: np.asarray(a, dtype=np.int32)
    x0 = [(7 * s) % 41 for s in range(n_shots)]
    x1 = [a + (115 if s % 3 else 140) for s, a in enumerate(x0)]
    rz, rx, off = [], [], [0]
    for s in range(n_shots):
        x = np.arange(x0[s], x1[s], 5)
        rx += list(x) + [x0[s]]  # two receivers share a cell
        rz += [(s + 11 * i) % nz for i in range(len(x))] + [s % nz]
        off.append(len(rx))
    g.src_iz = i32([(13 * s) % nz for s in range(n_shots)])
    g.src_ix = i32([x0[s] + (17 * s) % (x1[s] - x0[s]) for s in range(n_shots)])
    g.nt = i32([nt - s if s < n_shots // 2 else 1 + (37 * s) % nt for s in range(n_shots)])
    g.rec_off, g.rec_iz, g.rec_ix = i32(off), i32(rz), i32(rx)
    g.win_x0, g.win_x1 = i32(x0), i32(x1)
    c.geom = g
    tiles = sum(3 * -(-(b - a + 2 * nb) // 64) for a, b in zip(x0, x1))
    return c, v, tiles


# Tiles per resident CTA of the forward and adjoint kernels (two per SM; one per SM for
# Born of both fields): above one and below two (finished tiles published at once),
# and above two (published in the middle of the next tile).
@pytest.mark.parametrize("history", ["", "0", "1500"], ids=["history", "recompute", "partial"])
@pytest.mark.parametrize("n_shots,least,most", [(56, 1.0, 2.0), (130, 2.5, 9.0)], ids=["eager", "deferred"])
def test_many_pairs_equal_one_step(n_shots, least, most, history, monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c, v, tiles = _case(n_shots)
    ctas = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    assert least < tiles / ctas < most
    one = _run(c, v, False, history, monkeypatch)
    two = _run(c, v, True, history, monkeypatch)
    assert np.all(np.isfinite(one[0])) and all(np.linalg.norm(x) > 0 for x in one[:6])
    for a, b in zip(one, two):
        np.testing.assert_array_equal(a, b)


def test_launches_take_many_pairs(monkeypatch):
    """The form under test runs: a pass of 535 steps takes two launches and the
    model's preparation."""
    monkeypatch.setenv("DHFWI_STEP_VARIANT", "4")
    monkeypatch.setenv("DHFWI_TIME_BLOCK", "1")
    c, v, _ = _case(56)
    ctx = gpu_ctx(c)
    ctx.model_shots(to_dev(v), f32_geom(c.geom))
    assert ctx.stats()["kernel_launches"] == 3
    ctx.close()


def test_two_contexts_at_once():
    """Two threads, each with its own context and stream: the launches of one neither
    wait for nor disturb the other's."""
    import threading

    import torch

    c, v, _ = _case(56)
    g = f32_geom(c.geom)
    out = {}

    def work(k, rounds):
        ctx = gpu_ctx(c)
        with torch.cuda.stream(torch.cuda.Stream()):
            vd = to_dev(v)
            for _ in range(rounds):
                d = ctx.model_shots(vd, g)
                J, grad = ctx.fwi_gradient(vd, g, 0.5 * d)
                b = ctx.born_demig(vd, g, 0.01 * vd)
            torch.cuda.current_stream().synchronize()
            out[k] = [x.cpu().numpy() for x in (d, grad, b)] + [J]
        ctx.close()

    work("alone", 1)
    threads = [threading.Thread(target=work, args=(k, 3)) for k in ("a", "b")]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for k in ("a", "b"):
        for x, y in zip(out["alone"], out[k]):
            np.testing.assert_array_equal(x, y)
