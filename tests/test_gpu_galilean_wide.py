"""The Galilean walk over more coordinates than a warp has lanes: the first warp's loops over lanes and the
coordinate maps spread over warps by kind, against the oracle's walk (FP64, same stream).

The live set spreads by 0.02 around one point of the cube, so that some trials move, some reflect off the
contour and some off the walls.  Identical start points and move counts, end points to 1e-9 as in the narrower
walks' tests (a handful of steps of FP64 arithmetic on O(1) coordinates).
"""
import numpy as np
import pytest

import oracle
from helpers import event
from paper_1909_11873_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1909_11873_gb300 import build
    build.build()


@pytest.mark.parametrize("cfg,n_nodes", [("c1", 16), ("c2", 10)])  # 36 and 71 coordinates
def test_wide_galilean_replays_oracle_walk_fp64(cfg, n_nodes):
    from paper_1909_11873_gb300 import gwl

    ev = event(cfg)
    smp = ev.sampling
    nodes = I.cal_node_freqs(float(ev.freqs[0]), float(ev.freqs[-1]), n_nodes)
    n_cal = 2 * n_nodes * ev.n_det
    D, K = smp.D + n_cal, 96
    rng = np.random.default_rng(12)
    u = np.clip(0.5 + 0.02 * rng.standard_normal((K, D)), 0.001, 0.999)
    u[:, -1] = rng.uniform(0.001, 0.03, K)  # next to a wall
    cal = 0.1 * oracle.inv_normal_cdf(u[:, smp.D:]).reshape(K, n_cal)
    ll = oracle.loglike_cal(ev, nodes, np.concatenate([oracle.prior_transform(smp, u[:, :smp.D]), cal], axis=1))
    worst = int(np.argmin(ll))
    star = float(np.median(ll))
    chol = 0.02 * (np.eye(D) + 0.1 * np.tril(rng.standard_normal((D, D)), -1) / np.sqrt(D))
    n, wl, seed, ctr, scale = 12, 4, 0xCA2, 3, 0.2
    ctx = gwl.Context.from_event(ev, 0)
    ctx.gwl_set_calibration(nodes, 0.1, 0.1)
    ctx.gwl_set_walk(gwl.GWL_WALK_GALILEAN)
    ou = torch.zeros((n, D), dtype=torch.float64, device="cuda")
    ol = torch.zeros(n, dtype=torch.float64, device="cuda")
    on = torch.zeros(n, dtype=torch.int32, device="cuda")
    os_ = torch.zeros(n, dtype=torch.int32, device="cuda")
    ctx.ns_replace(torch.from_numpy(u).cuda(), torch.from_numpy(ll).cuda(), worst, star, seed, ctr, n, wl, scale,
                   torch.from_numpy(chol).cuda(), ou, ol, on, os_)
    torch.cuda.synchronize()
    ctx.gwl_sync()
    ru, rl, rn, rs = oracle.gmc_replace(ev, smp, u, ll, worst, star, seed, ctr, n, wl, scale, chol,
                                        cal=(nodes, 0.1, 0.1))
    assert np.array_equal(os_.cpu().numpy(), rs)
    assert np.array_equal(on.cpu().numpy(), rn)
    assert np.allclose(ou.cpu().numpy(), ru, rtol=0, atol=1e-9)
    assert np.allclose(ol.cpu().numpy(), rl, rtol=0, atol=1e-6)
    assert 0 < rn.sum() < n * wl
