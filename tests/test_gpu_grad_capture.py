"""The gradient recorded by a stream capture, beside eager calls on the same context."""
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
@pytest.mark.parametrize("with_cal", [False, True])
def test_recorded_call_vouches_for_nothing(precision, with_cal):
    """A gradient that a stream capture records has cleared no counters yet: an eager call before the first replay,
    the replay, and an eager call after it give what a fresh context gives.  The captured call is the context's first
    one (relaxed mode, so that it may allocate), then one whose window count has grown within the buffer's spare part."""
    from paper_1909_11873_gb300 import gwl as g

    ev = event("c1")
    B = 300
    rows = I.reduced(I.proposals(ev, 2 * B, 3), ev.sampling)
    if with_cal:
        rows = np.concatenate([rows, I.draw_calibration(np.random.default_rng(2), 2 * B, 1, 4)], axis=1)
    x, y = (torch.from_numpy(np.ascontiguousarray(r)).cuda() for r in (rows[:B], rows[B:]))

    def context():
        ctx = g.Context.from_event(ev, precision)
        if with_cal:
            ctx.gwl_set_calibration(I.cal_node_freqs(20.0, 512.0, 4))
        return ctx

    def fresh(window, rows):
        ctx = context()
        ctx.gwl_set_tuning(grad_window=window)
        out = g.grad(ctx, rows)
        ctx.gwl_sync()
        ctx.close()
        return out

    for eager_first, window in (((), 192), ((384, 256), 192)):
        # memory that the context's small buffers may be given is not clear
        junk = torch.full((1 << 22,), 0x5A5A5A5A, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        del junk
        torch.cuda.empty_cache()
        ctx = context()
        for w in eager_first:
            ctx.gwl_set_tuning(grad_window=w)
            g.grad(ctx, x)
        ctx.gwl_set_tuning(grad_window=window)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, capture_error_mode="relaxed"):
            rec = g.grad(ctx, x)
        eager = g.grad(ctx, y)
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        after = g.grad(ctx, y)
        ref_x, ref_y = fresh(window, x), fresh(window, y)
        for k in range(2):
            assert torch.equal(eager[k], ref_y[k]) and torch.equal(rec[k], ref_x[k]) and torch.equal(after[k], ref_y[k])
        ctx.gwl_sync()
        ctx.close()
