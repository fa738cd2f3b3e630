"""Stage 1 of the group-row dedispersion: groups of more rows than one pass of
records holds, rows that start at odd addresses and windows that end inside a
16-byte piece of the input, and short last groups.  The plane is bit-exact
against the CPU oracle."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


# the widest group has 421 rows at G = 4, 217 at G = 3, 72 at G = 2
@pytest.mark.parametrize("G", [2, 3, 4])
@pytest.mark.parametrize("nchan,nout", [(16, 4096), (17, 4083), (18, 9001), (16, 15)])
def test_many_rows_and_edges(G, nchan, nout, monkeypatch):
    from paper_2511_02328_gb300.search import Plan
    monkeypatch.setenv("AFGB_DEDISP_KERNEL", "pairs")
    monkeypatch.setenv("AFGB_PAIR_GROUP", str(G))
    dms, tsamp = np.arange(0.0, 1200.0, 1.0), 4e-3
    D = oracle.delay_table(nchan, 1000.0, 1500.0, tsamp, dms)
    nsamp = int(D.max()) + nout
    x = np.random.default_rng(nchan * nout).integers(0, 256, (nchan, nsamp), dtype=np.uint8)
    p = Plan(nchan, 1000.0, 1500.0, tsamp, dms)
    p.reserve(nsamp)
    assert p.kernel()["path"] == "pairs" and p.kernel()["group"] == G
    plane = p.dedisperse(torch.from_numpy(x).cuda())
    assert np.array_equal(plane.cpu().numpy(), oracle.dedisperse(x, D))
    p.close()
