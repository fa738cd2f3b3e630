"""The group-row sets' buffers at their limits: a stream's HBM budget holds as
many slots as the leanest set's buffer leaves, and a plan whose tables give a
larger set first still finds one within a small row budget."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


BAND, TSAMP = (1000.0, 1500.0), 1.9661e-4


def test_stream_slots_under_a_budget(monkeypatch):
    from paper_2511_02328_gb300 import _lib
    dms, widths, window = np.arange(0.0, 501.0, 1.0), [1, 4, 16], 1 << 16
    for k in ("AFGB_PAIR_GROUP", "AFGB_PAIR_DPW", "AFGB_DEDISP_KERNEL"):
        monkeypatch.delenv(k, raising=False)

    def slots(**env):
        for k, v in env.items():
            monkeypatch.setenv(k, v)
        h = _lib.af_stream_open(2, 1024, *BAND, TSAMP, dms, window, widths, 8.0, 4096, hbm_budget=4 << 30, max_slots=16)
        n = _lib.af_stream_info(h)[2]
        _lib.af_stream_close(h)
        for k in env:
            monkeypatch.delenv(k)
        return n

    # the leanest set of 15-row blocks is that of groups of 3 here
    assert slots() >= slots(AFGB_PAIR_GROUP="3", AFGB_PAIR_DPW="1") >= 1


@pytest.mark.parametrize("mb", [200, 600])
def test_small_row_budget(mb, monkeypatch):
    from paper_2511_02328_gb300.search import Plan
    monkeypatch.setenv("AFGB_PAIR_BUDGET_MB", str(mb))
    dms = np.arange(0.0, 301.0, 1.0)
    p = Plan(1024, *BAND, TSAMP, dms)
    x = torch.randint(0, 256, (1024, p.dmax + 20000), device="cuda", dtype=torch.uint8,
                      generator=torch.Generator(device="cuda").manual_seed(mb))
    a = p.dedisperse(x)
    monkeypatch.setenv("AFGB_DEDISP_KERNEL", "tile")
    q = Plan(1024, *BAND, TSAMP, dms)
    assert torch.equal(a, q.dedisperse(x))
    p.close()
    q.close()
