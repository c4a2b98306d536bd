"""The gradient's work counters stay cleared from call to call, whatever changes between calls.

Every sequence of window sizes, batch sizes, calibration on and off and likelihood calls in
between gives, call by call, what a fresh context gives bit for bit.
"""
import numpy as np
import pytest

from helpers import event
from paper_1909_11873_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1909_11873_gb300 import build

    build.build()


@pytest.mark.parametrize("precision", [0, 1])
def test_calls_do_not_see_each_other(precision):
    from paper_1909_11873_gb300 import gwl as g

    ev = event("c1")
    nodes = I.cal_node_freqs(20.0, 512.0, 4)
    th = I.reduced(I.proposals(ev, 700, 3), ev.sampling)
    th[7, 1] = 2.0  # an unphysical row
    cal = I.draw_calibration(np.random.default_rng(2), 700, 1, 4)

    def call(ctx, window, B, with_cal):
        ctx.gwl_set_calibration(nodes if with_cal else [])
        ctx.gwl_set_tuning(grad_window=window)
        rows = np.concatenate([th, cal], axis=1) if with_cal else th
        return g.grad(ctx, torch.from_numpy(np.ascontiguousarray(rows[:B])).cuda())

    plan = [(384, 700, False), (128, 33, False), (128, 700, False), (384, 1, True), (256, 700, True), (128, 64, True),
            (384, 700, False), (384, 700, False)]
    one = g.Context.from_event(ev, precision)
    for k, (window, B, with_cal) in enumerate(plan):
        got = call(one, window, B, with_cal)
        if k % 3 == 1:  # a likelihood call in between
            g.loglike(one, torch.from_numpy(np.ascontiguousarray(np.concatenate([th, cal], axis=1) if with_cal else th)).cuda())
        fresh = g.Context.from_event(ev, precision)
        ref = call(fresh, window, B, with_cal)
        for a, b in zip(got, ref):
            assert torch.equal(a, b), (k, window, B, with_cal)
        fresh.close()
    one.gwl_sync()
    one.close()
