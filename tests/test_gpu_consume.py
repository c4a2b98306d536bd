"""One round of the device sampler against the replacement loop written out in Python.

The live set comes from a checkpoint before the first round, the candidates from
ns_replace with the same seed, threshold and step matrix (Cholesky factor of the live
set's covariance, formed here: its rounding, 1e-13 of a coordinate, moves a log-likelihood
by less than the FP64 path's bar of 1e-6).  Sizes lie around the loop's own: fewer live
points than lanes, one candidate, the last size that one lane reads again and the first
that the warp does, more candidates than fit one register each.
"""
import numpy as np
import pytest

from helpers import event

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1909_11873_gb300 import build

    build.build()


@pytest.mark.parametrize("K,n", [(7, 3), (32, 1), (33, 70), (384, 129), (385, 200), (1100, 500)])
def test_round_matches_python_replacement_loop(K, n):
    from paper_1909_11873_gb300 import gwl as g

    ev = event("c1")
    ctx = g.Context.from_event(ev, g.GWL_FP64)
    D, walk, seed = ctx.n_dim, 4, 21
    cap = K + 2 * n
    st0 = ctx.ns_run(K, n, walk, seed, max_rounds=0, max_dead=cap, checkpoint=True)["state"]
    head = len(st0) - K * (D + 1) - cap * (D + 2)
    u, l = st0[head:head + K * D].reshape(K, D).copy(), st0[head + K * D:head + K * (D + 1)].copy()
    out = ctx.ns_run(K, n, walk, seed, max_rounds=1, max_dead=cap, checkpoint=True)
    worst = int(np.argmin(l))
    chol = np.linalg.cholesky(np.cov(u.T))
    cu = torch.empty((n, D), dtype=torch.float64, device="cuda")
    cl = torch.empty(n, dtype=torch.float64, device="cuda")
    cn = torch.empty(n, dtype=torch.int32, device="cuda")
    to = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    ctx.ns_replace(to(u), to(l), worst, l[worst], seed, 0, n, walk, 1.0, to(chol), cu, cl, cn)
    cu, cl = cu.cpu().numpy(), cl.cpu().numpy()
    dead_l, dead_u, live_l, live_u = [], [], l.copy(), u.copy()
    for c in range(n):
        k = int(np.argmin(live_l))
        if cl[c] > live_l[k]:
            dead_l.append(live_l[k])
            dead_u.append(live_u[k].copy())
            live_l[k], live_u[k] = cl[c], cu[c]
    m = len(dead_l)
    assert out["n_dead"] == m + K
    np.testing.assert_allclose(out["dead_lnl"][:m], dead_l, rtol=0, atol=1e-6)
    np.testing.assert_allclose(out["dead_u"][:m], np.array(dead_u).reshape(m, D), rtol=0, atol=1e-9)
    s1 = out["state"]
    np.testing.assert_allclose(s1[head + K * D:head + K * (D + 1)], live_l, rtol=0, atol=1e-6)
    np.testing.assert_allclose(s1[head:head + K * D].reshape(K, D), live_u, rtol=0, atol=1e-9)
    ctx.close()
