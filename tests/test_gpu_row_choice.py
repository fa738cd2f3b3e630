"""Which kernel a plan gets by default: group rows or channel tiles by one
comparison of both predicted times, blocks of 15 and of 30 DM rows each where it is
predicted faster, and rows in several blocks within a small budget; the planes and
row sums are those of the plan forced onto channel tiles."""
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
    for k in ("AFGB_DEDISP_KERNEL", "AFGB_PAIR_GROUP", "AFGB_PAIR_DPW", "AFGB_PAIR_STAGES", "AFGB_PAIR_BUDGET_MB"):
        monkeypatch.delenv(k, raising=False)


def _run(p, x):
    stats = torch.empty((p.ndm, 2), dtype=torch.int64, device="cuda")
    return p.dedisperse(x, stats=stats), stats


def _check(monkeypatch, nchan, ndm, nout, **env):
    """(kernel, row bytes of one call, of the buffer) of the default plan, after comparing it with channel tiles."""
    from paper_2511_02328_gb300 import _lib
    from paper_2511_02328_gb300.search import Plan
    dms = np.arange(ndm) * 1.0
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    p = Plan(nchan, *BAND, TSAMP, dms)
    nsamp = p.dmax + nout
    x = torch.randint(0, 256, (nchan, nsamp), device="cuda", dtype=torch.uint8,
                      generator=torch.Generator(device="cuda").manual_seed(nchan + ndm))
    p.reserve(nsamp)
    k = p.kernel()
    size = _lib.af_dedisperse_workspace_size(p.handle, nsamp)
    if k["path"] == "pairs":
        _lib.af_dedisperse_timing(p.handle, 1)
    plane, stats = _run(p, x)
    rows = _lib.af_dedisperse_times(p.handle, 0)[2] if k["path"] == "pairs" else 0
    monkeypatch.setenv("AFGB_DEDISP_KERNEL", "tile")
    q = Plan(nchan, *BAND, TSAMP, dms)
    ref, ref_stats = _run(q, x)
    assert q.kernel()["path"] == "tile" and torch.equal(plane, ref) and torch.equal(stats, ref_stats)
    p.close()
    q.close()
    monkeypatch.delenv("AFGB_DEDISP_KERNEL")
    return k, rows, size


# both sides of the line, by a factor of 1.4 and more in measured time
@pytest.mark.parametrize("nchan,ndm,nout,path", [(128, 1001, 5000, "tile"), (64, 400, 150000, "tile"), (16, 16, 5000, "tile"),
                                                 (4096, 16, 700, "pairs"), (1024, 4, 5000, "pairs"),
                                                 (1024, 301, 60000, "pairs"), (512, 128, 30000, "pairs")])
def test_rows_or_tiles(nchan, ndm, nout, path, monkeypatch):
    k, _, size = _check(monkeypatch, nchan, ndm, nout)
    assert k["path"] == path and (size > 0) == (path == "pairs")


def test_both_block_heights_are_picked(monkeypatch):
    from paper_2511_02328_gb300.search import Plan
    nchan, ndm = 1024, 301
    heights = {}
    for nout in (8000, 20000, 60000):
        k, _, _ = _check(monkeypatch, nchan, ndm, nout)
        for dpw in (1, 2):
            monkeypatch.setenv("AFGB_PAIR_DPW", str(dpw))
            monkeypatch.setenv("AFGB_PAIR_GROUP", str(k["group"]))
            f = Plan(nchan, *BAND, TSAMP, np.arange(ndm) * 1.0)
            f.reserve(f.dmax + nout)
            if f.kernel()["spread"] == k["spread"]:  # a block of 30 rows spans more delays
                heights[nout] = dpw
            f.close()
            monkeypatch.delenv("AFGB_PAIR_DPW")
            monkeypatch.delenv("AFGB_PAIR_GROUP")
    assert len(heights) == 3 and set(heights.values()) == {1, 2}


@pytest.mark.parametrize("mb", [200, 600])
def test_small_budget_runs_several_blocks_of_rows(mb, monkeypatch):
    k, rows, size = _check(monkeypatch, 1024, 301, 60000, AFGB_PAIR_BUDGET_MB=str(mb))
    assert k["path"] == "pairs" and 0 < size <= mb << 20 < rows
