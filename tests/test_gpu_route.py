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


def test_first_calls_under_capture():
    """Calls that take the separate kernels, although they fit the one-kernel form, need scratch; recorded as a
    context's first calls, when nothing may be allocated, they take the one-kernel form instead."""
    from paper_1909_11873_gb300 import gwl as g

    ev = custom_event(dict(n_det=3, T=32.0, f_low=20.0, f_high=1024.0, noise=True, source="bns", gmst=1.7), 9)
    dims = [I.IDX["psi"], I.IDX["ra"], I.IDX["tc"], I.IDX["phic"]]
    smp = I.Sampling(np.array(dims, dtype=np.int32), ev.theta_inj.copy(), np.zeros(4, dtype=np.int32), np.zeros(4),
                     np.ones(4), np.array([1, 0, 0, 1], dtype=np.int32))
    rng = np.random.default_rng(3)
    u = torch.from_numpy(rng.uniform(0.0, 1.0, (40, 4))).cuda()
    chol = torch.from_numpy(0.2 * np.eye(4)).cuda()
    n = 3

    def context():
        ctx = g.Context.from_event(ev, g.GWL_MIXED, sampling=smp)
        ctx.gwl_set_tuning(window=1280, bin_kernel=g.GWL_BINS_WARP)
        return ctx

    def calls(ctx, l, star, out):
        lnl = g.loglike(ctx, u[:n])
        ctx.ns_replace(u, l, 0, star, 5, 1, n, 4, 0.5, chol, *out)
        return lnl

    def outputs():
        return [torch.zeros((n, 4), dtype=torch.float64, device="cuda"), torch.zeros(n, dtype=torch.float64, device="cuda"),
                torch.zeros(n, dtype=torch.int32, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda")]

    eager = context()
    k = eager.launch_count()
    l = g.loglike(eager, u)
    assert eager.launch_count() - k == 3  # (such a call: few rows of many groups of windows)
    star = float(l.min()) - 1.0
    want = outputs()
    k = eager.launch_count()
    ref = calls(eager, l, star, want)
    assert eager.launch_count() - k > 4  # (so is the walk)
    ctx = context()
    out, graph = outputs(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        lnl = calls(ctx, l, star, out)
    graph.replay()
    torch.cuda.synchronize()
    assert float((lnl - ref).abs().max()) < 1e-10
    assert torch.equal(out[2], want[2]) and torch.equal(out[3], want[3]) and torch.equal(out[0], want[0])
    assert float((out[1] - want[1]).abs().max()) < 1e-10
    # the graph holds no scratch: it gives the same after calls that have replaced the context's
    first = [lnl.clone()] + [o.clone() for o in out]
    for rows in (u, u.repeat(100, 1)):
        g.loglike(ctx, rows)
    g.grad(ctx, u.repeat(100, 1))
    graph.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(first, [lnl] + out))
    ctx.gwl_sync()
