"""The one-kernel likelihood against the separate prologue and bin-loop kernels.

With the largest windows a batch of more than eight rows per SM does not fit the
one-kernel form and takes the separate kernels (three launches), while the same
rows in smaller calls take the one-kernel form (one launch).  Both add the
same FP32 terms in the same order within a window, so rows with one window are
equal bit for bit; with several windows the FP64 sums over windows may be added
in another order: up to 32 window sums of a few hundred, 32 * 2^-53 * 1e4 < 1e-10.
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


def launches(ctx, fn):
    n = ctx.launch_count()
    out = fn()
    return out, ctx.launch_count() - n


@pytest.mark.parametrize("n_det,T,source,fcut,nodes", [
    (1, 4.0, "bbh", 0, 0),   # one window, short rows
    (3, 8.0, "bbh", 0, 0),
    (4, 8.0, "bbh", 0, 3),   # calibration model, four detectors
    (3, 8.0, "bbh", 1, 10),  # every row in every window, windows in several groups
    (2, 8.0, "bns", 0, 0),   # float-float deltas at low frequency, ragged last window
])
def test_one_kernel_matches_separate_kernels(n_det, T, source, fcut, nodes):
    from paper_1909_11873_gb300 import gwl as g

    cfg = dict(n_det=n_det, T=T, f_low=20.0, f_high=1024.0, noise=True, source=source, gmst=1.7)
    ev = custom_event(cfg, 3, fcut_mode=fcut)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 8 * sms + 35
    th = I.reduced(I.proposals(ev, n, 9), ev.sampling)
    th[5, 1] = 1.5       # unphysical rows, alone and at a group's end
    th[-1, 0] = np.nan
    th[31, 0] = 400.0    # without an in-band bin where the cut is the ISCO's
    if nodes:
        th = np.concatenate([th, I.draw_calibration(np.random.default_rng(4), n, n_det, nodes)], axis=1)
    x = torch.from_numpy(np.ascontiguousarray(th)).cuda()
    ctx = g.Context.from_event(ev, g.GWL_MIXED)
    if nodes:
        ctx.gwl_set_calibration(I.cal_node_freqs(20.0, 1024.0, nodes))
    window = 1344 if n_det == 4 else 1440 if nodes else 1696 if n_det == 3 else 2432  # the largest that is accepted
    ctx.gwl_set_tuning(window=window, ctas_per_sm=2, bin_kernel=g.GWL_BINS_WARP)
    ref, k = launches(ctx, lambda: g.loglike(ctx, x))
    assert k == 3, "the reference is meant to take the separate kernels"
    for sizes in ([1, 2, 7, 8, 9, 31, 32, 33, 152, 153], [sms, 8 * sms - sms - 428]):
        a = 0
        for B in sizes:
            got, k = launches(ctx, lambda: g.loglike(ctx, x[a:a + B].contiguous()))
            assert k == 1
            r = ref[a:a + B]
            assert torch.equal(torch.isinf(got), torch.isinf(r))
            d = (got - r)[~torch.isinf(r)].abs()
            if fcut == 0 and source == "bbh":
                assert torch.equal(got, r), f"B={B}: {float(d.max()):.3e}"
            else:
                assert float(d.max()) < 1e-10, f"B={B}: {float(d.max()):.3e}"
            a += B
    got = torch.cat([g.loglike(ctx, x[-40:].contiguous())])  # the batch's end, NaN row last
    assert torch.equal(torch.isinf(got), torch.isinf(ref[-40:]))
    # whole waves of two CTAs per SM, and the same rows whatever the batch they come in
    ctx.gwl_set_tuning(window=640)
    one = torch.cat([g.loglike(ctx, x[a:a + 100].contiguous()) for a in range(0, n, 100)])
    many, k = launches(ctx, lambda: g.loglike(ctx, x.repeat(9, 1)))
    assert k == 1
    assert torch.equal(many.reshape(9, n), one[None].expand(9, n))
    ctx.gwl_sync()
    ctx.close()


@pytest.mark.parametrize("n_det,source,nodes,walk", [(1, "bbh", 0, 6), (3, "bbh", 0, 5), (3, "bbh", 10, 3), (2, "bbh", 0, 0)])
def test_one_kernel_walk_matches_separate_kernels(n_det, source, nodes, walk):
    """Chain b's random numbers depend on b alone, so the first chains of a long batch (separate kernels, with the
    largest windows) are those of a short one (one kernel): same points, acceptances and, rows having one window,
    the same log-likelihoods bit for bit."""
    from paper_1909_11873_gb300 import gwl as g

    cfg = dict(n_det=n_det, T=8.0, f_low=20.0, f_high=1024.0, noise=True, source=source, gmst=1.7)
    ev = custom_event(cfg, 5)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ctx = g.Context.from_event(ev, g.GWL_MIXED)
    if nodes:
        ctx.gwl_set_calibration(I.cal_node_freqs(20.0, 1024.0, nodes))
    ctx.gwl_set_tuning(window=1440 if nodes else 1696 if n_det == 3 else 2432, bin_kernel=g.GWL_BINS_WARP)
    D, K = ctx.theta_stride, 64
    rng = np.random.default_rng(8)
    u = torch.from_numpy(rng.uniform(0.0, 1.0, (K, D))).cuda()
    l = torch.from_numpy(np.sort(rng.uniform(-50.0, 0.0, K))).cuda()
    A = 0.1 * np.tril(rng.standard_normal((D, D))) / np.sqrt(D) + 0.05 * np.eye(D)
    chol = torch.from_numpy(A).cuda()

    def chains(n):
        out = [torch.empty((n, D), dtype=torch.float64, device="cuda"), torch.empty(n, dtype=torch.float64, device="cuda"),
               torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda")]
        k = ctx.launch_count()
        ctx.ns_replace(u, l, 0, -200.0, 7, 3, n, walk, 0.5, chol, *out)
        torch.cuda.synchronize()
        return out, ctx.launch_count() - k

    ref, k = chains(8 * sms + 9)
    assert walk == 0 or (k > 1 and int((ref[2] > 0).sum()) > 0)
    for n in (1, 9, sms + 1, 8 * sms):
        got, k = chains(n)
        assert k == 1
        for a, b in zip(got, ref):
            assert torch.equal(a, b[:n])
    ctx.gwl_sync()
    ctx.close()


@pytest.mark.parametrize("n_det,T,source,fcut", [(3, 8.0, "bbh", 0), (1, 4.0, "bbh", 0), (4, 4.0, "bns", 1), (2, 16.0, "bbh", 0)])
def test_one_kernel_fp64_at_every_shape(n_det, T, source, fcut):
    """The FP64 one-kernel form at the batch sizes where its shape changes (clusters of eight, four and two CTAs,
    one CTA per group, 32 rows, two waves) against one batch in another shape: on the 16 s segment the separate
    kernels.  FP64 sums in another order: about 1e4 terms of up to 10 each, 1e4 * 2^-53 * 1e3 < 2e-9."""
    from paper_1909_11873_gb300 import gwl as g

    cfg = dict(n_det=n_det, T=T, f_low=20.0, f_high=1024.0, noise=True, source=source, gmst=1.7)
    ev = custom_event(cfg, 4, fcut_mode=fcut)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 8 * sms - 1
    th = I.reduced(I.proposals(ev, n, 10), ev.sampling)
    th[5, 1] = 1.5
    th[-1, 0] = np.nan
    th[31, 0] = 400.0
    x = torch.from_numpy(th).cuda()
    ctx = g.Context.from_event(ev, g.GWL_FP64)
    ref, k = launches(ctx, lambda: g.loglike(ctx, x))
    assert k == (3 if T == 16.0 else 1)
    ok = ~torch.isinf(ref)
    sizes = [1, 2, sms * 2 // 19, sms * 2 // 19 + 1, sms * 4 // 19 + 1, sms // 2, sms // 2 + 1, sms, sms + 1, 2 * sms, 2 * sms + 1]
    for B in sizes if T != 16.0 else []:
        got, k = launches(ctx, lambda: g.loglike(ctx, x[:B].contiguous()))
        again = g.loglike(ctx, x[:B].contiguous())
        assert k == 1 and torch.equal(got, again)
        assert torch.equal(torch.isinf(got), ~ok[:B])
        d = (got - ref[:B])[ok[:B]].abs()
        assert d.numel() == 0 or float(d.max()) < 2e-9, f"B={B}: {float(d.max()):.3e}"
    for times in (2, 5, 33):  # from a row per warp to two waves of 32 rows per SM
        got, k = launches(ctx, lambda: g.loglike(ctx, x.repeat(times, 1)[: times * n if times < 33 else 32 * sms + 5]))
        assert k == (3 if T == 16.0 else 1)
        want = ref.repeat(times)[: got.numel()]
        assert torch.equal(torch.isinf(got), torch.isinf(want))
        assert float((got - want)[~torch.isinf(want)].abs().max()) < 2e-9
    ctx.gwl_sync()
    ctx.close()
