"""Rows of a multi-event batch that share a warp's table reads.

A row's sums take its own blocks in their own order, whichever rows it shares a
warp with, so its lnL is the same bits in every batch it appears in: batches of
sizes around the warps' and the tasks' row counts are compared with one row at a
time and with a reversed batch.
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


@pytest.mark.parametrize("n_det,T,source,fcut", [
    (1, 4.0, "bbh", 0),    # short rows of all lengths: few blocks in common
    (2, 32.0, "bns", 0),   # float-float blocks before the shared ones, many windows
    (3, 8.0, "bbh", 1),    # every row complete in every window
    (4, 8.0, "bns", 0),    # tasks of 32 rows
])
def test_rows_do_not_depend_on_their_neighbours(n_det, T, source, fcut):
    from paper_1909_11873_gb300 import gwl as g

    evs = [custom_event(dict(n_det=n_det, T=t, f_low=20.0, f_high=1024.0, noise=True, source=source, gmst=1.7), 3,
                        fcut_mode=fcut) for t in (T, 4.0)]
    n = 67
    rows = [I.reduced(I.proposals(ev, n, 9 + i), ev.sampling) for i, ev in enumerate(evs)]
    rows[0][5, 1] = 1.5       # an unphysical row
    rows[0][31, 0] = 400.0    # without an in-band bin where the cut is the ISCO's
    ctxs = [g.Context.from_event(ev, g.GWL_MIXED) for ev in evs]
    mc = g.MultiContext(ctxs)

    def run(pick):
        x = torch.from_numpy(np.ascontiguousarray(np.concatenate([r[pick] for r in rows]))).cuda()
        out = torch.empty(x.shape[0], dtype=torch.float64, device="cuda")
        mc.gwl_multi_loglike(x, out)
        return out.cpu().numpy().reshape(2, -1)

    one = np.concatenate([run(np.array([i])) for i in range(n)], axis=1)
    assert one[0, 5] == -np.inf and np.isfinite(np.delete(one[0], 5)).all()
    for k in (2, 3, 4, 5, 33, 63, 64, 65, 67):
        assert np.array_equal(run(np.arange(k)), one[:, :k]), k
    assert np.array_equal(run(np.arange(n)[::-1]), one[:, ::-1])
