"""The row sets a plan does not use: their tables leave the host's memory with the
first reservation, and a later reservation that picks another set builds that
set's tables again, to the same plane."""
import ctypes
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BAND, TSAMP = (1000.0, 1500.0), 2e-4


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.fixture(autouse=True)
def _default_choice(monkeypatch):
    for k in ("AFGB_PAIR_GROUP", "AFGB_PAIR_DPW", "AFGB_PAIR_STAGES", "AFGB_PAIR_BUDGET_MB"):
        monkeypatch.delenv(k, raising=False)
    monkeypatch.setenv("AFGB_DEDISP_KERNEL", "pairs")  # rows even where channel tiles are faster


def test_growing_lengths_switch_sets(monkeypatch):
    from paper_2511_02328_gb300 import _lib
    from paper_2511_02328_gb300.search import Plan
    nchan, dms = 512, np.arange(609) * 1.0
    p, t = Plan(nchan, *BAND, TSAMP, dms), Plan(nchan, *BAND, TSAMP, dms)
    x = torch.randint(0, 256, (nchan, p.dmax + 20000), device="cuda", dtype=torch.uint8,
                      generator=torch.Generator(device="cuda").manual_seed(2))
    ref = torch.empty((t.ndm, 20000), dtype=torch.int32, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    _lib.af_dedisperse(t.handle, x.data_ptr(), x.shape[1], ref.data_ptr(), 0, s)  # nothing reserved: channel tiles
    monkeypatch.setenv("AFGB_PAIR_STAGES", "4")  # read when the plan was made, not when a set is built again
    monkeypatch.setenv("AFGB_PAIR_BUDGET_MB", "1")
    seen = []
    for nout in (2000, 8000, 20000):
        xs = x[:, :p.dmax + nout].contiguous()
        plane = p.dedisperse(xs)
        assert torch.equal(plane, ref[:, :nout])
        seen.append(p.kernel())
    assert all(k["path"] == "pairs" and k["ring"] == 3 for k in seen)
    assert len({(k["group"], k["spread"]) for k in seen}) == 3  # three sets, one after another
    p.close()
    t.close()


def _rss():
    ctypes.CDLL(None).malloc_trim(0)
    return int(open("/proc/self/statm").read().split()[1]) * os.sysconf("SC_PAGE_SIZE")


def test_host_memory_of_reserved_plans():
    from paper_2511_02328_gb300.search import Plan
    def plan():
        p = Plan(2048, *BAND, TSAMP, np.arange(609) * 1.0)
        p.reserve(p.dmax + 4000)
        return p
    plans = [plan()]
    before = _rss()
    plans += [plan() for _ in range(6)]
    per_plan = (_rss() - before) / 6
    print("%.1f MB a plan" % (per_plan / 1e6))
    # kept: delays (5 MB), windows of the used set (8 bytes each), rows of six sets (24 bytes each)
    assert per_plan < 20e6
    for p in plans:
        p.close()
