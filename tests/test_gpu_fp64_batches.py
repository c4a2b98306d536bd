"""A row's FP64 log-likelihood has the same bits in every batch.

The one-kernel form chooses its rows and CTAs per group by the batch; the order of a row's sums does not follow them.
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


@pytest.mark.parametrize("n_det,T,f_high,source,fcut", [
    (3, 8.0, 1024.0, "bbh", 0),
    (1, 4.0, 512.0, "bbh", 0),
    (4, 8.0, 1023.0, "bns", 1),  # every row over the whole band, more pieces than a CTA stages together
    (2, 1.0, 83.0, "bbh", 1),    # one piece, and one lane of a second
])
def test_rows_do_not_depend_on_their_batch(n_det, T, f_high, source, fcut):
    from paper_1909_11873_gb300 import gwl as g

    cfg = dict(n_det=n_det, T=T, f_low=20.0, f_high=f_high, noise=True, source=source, gmst=1.7)
    ev = custom_event(cfg, 6, fcut_mode=fcut)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 2 * sms + 1
    th = I.reduced(I.proposals(ev, n, 12), ev.sampling)
    th[5, 1] = 1.5
    x = torch.from_numpy(th).cuda()
    ctx = g.Context.from_event(ev, g.GWL_FP64)
    ref = g.loglike(ctx, x)
    # clusters of eight, four and two CTAs, single CTAs, 32 rows per CTA, two waves
    sizes = [1, 2, sms * 2 // 19, sms * 2 // 19 + 1, sms * 4 // 19 + 1, sms // 2, sms // 2 + 1, sms, sms + 1]
    for B in sizes:
        for a in (0, n - B):
            assert torch.equal(g.loglike(ctx, x[a:a + B].contiguous()), ref[a:a + B]), (B, a)
    for times in (3, 17) if fcut else (3, 17, 33):
        assert torch.equal(g.loglike(ctx, x.repeat(times, 1)), ref.repeat(times)), times
    ctx.gwl_sync()
    ctx.close()
