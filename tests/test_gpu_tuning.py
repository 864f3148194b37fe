"""What the autotuner of a first call at a geometry leaves behind: the statistics of
the call itself, and trials that follow from the records alone."""
import copy

import numpy as np
import pytest

import synth
from gpu_helpers import f32, f32_geom, gpu_ctx, to_dev

pytestmark = pytest.mark.gpu


def _case(monkeypatch, nt=40, nt_max=None):
    for k in ("DHFWI_STEP_VARIANT", "DHFWI_TIME_BLOCK", "DHFWI_HISTORY_MB"):
        monkeypatch.delenv(k, raising=False)
    c = synth.tiny_case(nz=60, nx=90, nt=nt_max or nt, nb=20, n_shots=2, seed=3)
    c.geom.nt = np.full_like(c.geom.nt, nt)
    v = to_dev(f32(1800.0 + 400.0 * synth.rng(7).uniform(size=(60, 90))))
    return c, f32_geom(copy.deepcopy(c.geom)), v


def test_first_call_counts_its_own_updates(monkeypatch):
    c, g, v = _case(monkeypatch)
    for call in ("model", "gradient", "born"):
        ctx = gpu_ctx(c)
        cells = []
        for _ in range(2):
            if call == "model":
                ctx.model_shots(v, g)
            elif call == "gradient":
                ctx.fwi_gradient(v, g, ctx.new_data(g).zero_())
            else:
                ctx.born_demig(v, g, 0.01 * v)
            cells.append(ctx.stats()["cell_updates"])
        ctx.close()
        w = g.win_x1.astype(np.int64) - g.win_x0 + 2 * c.nb
        once = int(np.sum(w * g.nt)) * (c.nz + 2 * c.nb)
        assert cells == [(1 if call == "model" else 2) * once] * 2, call


def test_trials_follow_the_records(monkeypatch):
    """Records far shorter than the geometry's nt_max (its wavelets' length): the
    trials are those of a geometry whose nt_max is the longest record."""
    extra = []
    for nt_max in (6, 60):
        c, g, v = _case(monkeypatch, nt=6, nt_max=nt_max)
        ctx = gpu_ctx(c)
        launches = []
        for _ in range(2):
            ctx.model_shots(v, g)
            launches.append(ctx.stats()["kernel_launches"])
        extra.append(launches[0] - launches[1])
        ctx.close()
    assert extra[0] == extra[1]


def test_born_is_tried_by_the_first_born_call(monkeypatch):
    """Programs that never call Born don't pay for its trials; those that do pay once,
    whichever call came first."""
    c, g, v = _case(monkeypatch)

    def launches(calls):
        ctx = gpu_ctx(c)
        out = []
        for call in calls:
            if call == "model":
                ctx.model_shots(v, g)
            else:
                ctx.born_demig(v, g, 0.01 * v)
            out.append(ctx.stats()["kernel_launches"])
        ctx.close()
        return out

    m0, m1, b0, b1 = launches(["model", "model", "born", "born"])
    c0, c1, n0, n1 = launches(["born", "born", "model", "model"])
    assert m0 > m1 and b0 > b1
    assert c0 - c1 == (m0 - m1) + (b0 - b1)
    assert n0 == n1


def test_a_depth_is_not_fixed_by_one_sample(monkeypatch):
    """Every depth trial runs once for warm-up and is timed twice: for Born on a plan
    of one pair per launch three times four launches of both fields, four of the
    scattered field from the history and eight single steps of it."""
    c, g, v = _case(monkeypatch)
    ctx = gpu_ctx(c)
    ctx.model_shots(v, g)
    launches = []
    for _ in range(2):
        ctx.born_demig(v, g, 0.01 * v)
        launches.append(ctx.stats()["kernel_launches"])
    ctx.close()
    assert launches[0] - launches[1] == 3 * (4 + 4 + 8)
