"""Which calls of the mixed likelihood take one kernel, and that both forms agree across that line.

Window sums are the same in both forms; the FP64 sums over up to 26 windows of at most 1e4 each may be added in another
order: 26 * 1e4 * 2^-53 < 1e-10.
"""
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


@pytest.mark.parametrize("n_det,T,source,fcut,nodes,window,few,many", [
    (3, 8.0, "bbh", 0, 0, 640, 1, 1),    # short rows: one kernel at any batch
    (3, 32.0, "bbh", 0, 0, 1280, 1, 1),  # rows short of a long segment
    (2, 16.0, "bbh", 1, 0, 640, 1, 1),
    (3, 16.0, "bns", 0, 0, 1280, 3, 1),  # a row's windows in many groups: few rows spread over the chip
    (3, 32.0, "bns", 0, 0, 1280, 3, 1),
    (3, 16.0, "bns", 0, 10, 640, 3, 1),  # calibrated
])
def test_long_rows_in_small_batches_take_the_separate_kernels(n_det, T, source, fcut, nodes, window, few, many):
    from paper_1909_11873_gb300 import gwl as g

    ev = custom_event(dict(n_det=n_det, T=T, f_low=20.0, f_high=1024.0, noise=True, source=source, gmst=1.7), 9, fcut_mode=fcut)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 16 * sms
    th = I.reduced(I.proposals(ev, n, 14), ev.sampling)
    if nodes:
        th = np.concatenate([th, I.draw_calibration(np.random.default_rng(4), n, n_det, nodes)], axis=1)
    x = torch.from_numpy(np.ascontiguousarray(th)).cuda()
    ctx = g.Context.from_event(ev, g.GWL_MIXED)
    if nodes:
        ctx.gwl_set_calibration(I.cal_node_freqs(20.0, 1024.0, nodes))
    ctx.gwl_set_tuning(window=window, bin_kernel=g.GWL_BINS_WARP)

    def call(rows):
        k = ctx.launch_count()
        out = g.loglike(ctx, rows)
        return out, ctx.launch_count() - k

    ref, k = call(x)
    assert k == many
    for B in (1, 2, 17):
        got, k = call(x[:B].contiguous())
        assert k == few
        assert float((got - ref[:B]).abs().max()) < 1e-10
    ctx.gwl_sync()
    ctx.close()
