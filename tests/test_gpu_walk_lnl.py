"""The walks' log-likelihoods are gwl_loglike's, bit for bit.

The sampled coordinates have the prior U(0, 1), whose map is exact, so a chain's end point is also its parameter row:
where a chain has moved, the lnL that the walk carries is that of a gwl_loglike batch of the end points.
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


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n_det,T,source,fcut", [
    (3, 8.0, "bbh", 0),   # rows that end in the first window
    (1, 4.0, "bbh", 0),
    (3, 8.0, "bns", 0),   # float-float deltas; the windows in several groups, staged again at each step
    (2, 16.0, "bbh", 1),  # 26 windows, the last one ragged; FP64 in the separate kernels
])
def test_walk_carries_the_likelihoods_of_its_points(precision, n_det, T, source, fcut):
    from paper_1909_11873_gb300 import gwl as g

    cfg = dict(n_det=n_det, T=T, f_low=20.0, f_high=1024.0, noise=True, source=source, gmst=1.7)
    ev = custom_event(cfg, 7, fcut_mode=fcut)
    dims = [I.IDX["psi"], I.IDX["ra"], I.IDX["tc"], I.IDX["phic"]]
    D = len(dims)
    smp = I.Sampling(np.array(dims, dtype=np.int32), ev.theta_inj.copy(), np.zeros(D, dtype=np.int32), np.zeros(D),
                     np.ones(D), np.array([1, 0, 0, 1], dtype=np.int32))
    ctx = g.Context.from_event(ev, precision, sampling=smp)
    K = 60
    rng = np.random.default_rng(11)
    live_u = torch.from_numpy(rng.uniform(0.0, 1.0, (K, D))).cuda()
    live_l = g.loglike(ctx, live_u)
    worst = int(torch.argsort(live_l)[K // 3])
    chol = torch.from_numpy(np.tril(rng.uniform(-0.1, 0.1, (D, D))) + 0.15 * np.eye(D)).cuda()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for n in (1, 9, sms + 1, 8 * sms + 9, 2047, 2048):
        u, l = torch.empty((n, D), dtype=torch.float64, device="cuda"), torch.empty(n, dtype=torch.float64, device="cuda")
        acc, start = (torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(2))
        ctx.ns_replace(live_u, live_l, worst, float(live_l[worst]), 5, n, n, 3, 0.7, chol, u, l, acc, start)
        moved = acc > 0
        assert torch.equal(l[moved], g.loglike(ctx, u)[moved]), n
        assert torch.equal(l[~moved], live_l[start.long()][~moved])
        assert torch.equal(u[~moved], live_u[start.long()][~moved])
        assert n < 9 or 0 < int(moved.sum()) and bool((l[moved] >= live_l[worst]).all())
    ctx.gwl_sync()
    ctx.close()
