"""Device memory of a context: the blocked tables of the mixed path are held by mixed contexts only."""
import pytest

from helpers import custom_event

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1909_11873_gb300 import build

    build.build()


@pytest.mark.parametrize("n_det,units", [(1, 3), (2, 3), (3, 4), (4, 4)])
def test_blocked_tables_in_mixed_contexts_only(n_det, units):
    from paper_1909_11873_gb300 import gwl as g

    ev = custom_event(dict(n_det=n_det, T=4.0, f_low=20.0, f_high=523.0, noise=True, source="bbh", gmst=1.7), 8)
    size = {p: g.Context.from_event(ev, p).device_bytes() for p in (g.GWL_FP64, g.GWL_MIXED, g.GWL_MIXED_F64PHASE)}
    blocks = -(-ev.M // 32)
    assert size[g.GWL_MIXED] - size[g.GWL_FP64] == blocks * 32 * 16 * (units + 2)  # 16-byte units of a bin, low parts
    assert size[g.GWL_MIXED_F64PHASE] == size[g.GWL_FP64]
