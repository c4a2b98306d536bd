"""The autotuner leaves alone what the kernel that a batch takes does not read."""
import numpy as np
import pytest

from helpers import custom_event
from paper_1909_11873_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1909_11873_gb300 import build

    build.build()


@pytest.mark.parametrize("precision,T,nodes", [(0, 8.0, 0), (0, 16.0, 0), (1, 8.0, 0), (1, 8.0, 10)])
def test_unread_settings_are_not_tuned(precision, T, nodes):
    from paper_1909_11873_gb300 import gwl as g

    ev = custom_event(dict(n_det=3, T=T, f_low=20.0, f_high=1024.0, noise=True, source="bbh", gmst=1.7), 8)
    B = 300
    rows = I.reduced(I.proposals(ev, B, 4), ev.sampling)
    if nodes:
        rows = np.concatenate([rows, I.draw_calibration(np.random.default_rng(1), B, 3, nodes)], axis=1)
    ctx = g.Context.from_event(ev, precision)
    if nodes:
        ctx.gwl_set_calibration(I.cal_node_freqs(20.0, 1024.0, nodes))
    ctx.gwl_set_tuning(window=352, ctas_per_sm=2)  # a window that is no candidate
    x = torch.from_numpy(np.ascontiguousarray(rows)).cuda()
    n = ctx.launch_count()
    g.loglike(ctx, x)
    one_kernel = ctx.launch_count() - n == 1
    assert one_kernel == (precision == 1 or T == 8.0)
    t = ctx.gwl_autotune(x, what=g.GWL_TUNE_LOGLIKE)
    if precision == 0 and one_kernel:
        assert t["n_tried"] == 1 and t["window"] == 352
    if one_kernel and t["bin_kernel"] == g.GWL_BINS_WARP and t["window"] <= 1024:
        assert t["ctas_per_sm"] == 2
    if nodes or not one_kernel:  # no lane layout: a window is timed once where it takes one kernel, else with four grids
        want = 0
        for w in range(128, 1537, 64):
            try:
                ctx.gwl_set_tuning(window=w, bin_kernel=g.GWL_BINS_WARP)
            except g.GwlError:
                break
            n = ctx.launch_count()
            g.loglike(ctx, x)
            want += 1 if ctx.launch_count() - n == 1 else 4
        assert t["n_tried"] == want
    ctx.gwl_sync()
    ctx.close()
