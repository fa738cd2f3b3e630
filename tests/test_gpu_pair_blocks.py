"""Group-row dedispersion in blocks of 15 and of 30 DM rows (one or two per
consumer warp, the second's sums in tensor memory): plane and row sums
bit-exact against the CPU oracle for DM counts at the edges of a block, short
last groups, every ring depth, all-255 input (the largest 16-bit lane values
between folds), unsorted and repeated DMs, and several time blocks."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _check(monkeypatch, G, dpw, nchan, dms, nout, seed, full=False, ring=3, band=(1000.0, 1500.0), tsamp=2e-4):
    from paper_2511_02328_gb300.search import Plan
    monkeypatch.setenv("AFGB_DEDISP_KERNEL", "pairs")
    monkeypatch.setenv("AFGB_PAIR_GROUP", str(G))
    monkeypatch.setenv("AFGB_PAIR_DPW", str(dpw))
    monkeypatch.setenv("AFGB_PAIR_STAGES", str(ring))
    D = oracle.delay_table(nchan, band[0], band[1], tsamp, dms)
    nsamp = int(D.max()) + nout
    x = np.full((nchan, nsamp), 255, np.uint8) if full else \
        np.random.default_rng(seed).integers(0, 256, (nchan, nsamp), dtype=np.uint8)
    p = Plan(nchan, band[0], band[1], tsamp, dms)
    p.reserve(nsamp)
    k = p.kernel()
    assert (k["path"], k["group"], k["ring"]) == ("pairs", G, ring)
    stats = torch.empty((p.ndm, 2), dtype=torch.int64, device="cuda")
    plane = p.dedisperse(torch.from_numpy(x).cuda(), stats=stats)
    torch.cuda.synchronize()
    Y = oracle.dedisperse(x, D)
    assert np.array_equal(plane.cpu().numpy(), Y)
    S, Q = oracle.rowstats(Y)
    st = stats.cpu().numpy()
    assert np.array_equal(st[:, 0], S) and np.array_equal(st[:, 1], Q)
    p.close()


@pytest.mark.parametrize("dpw", [1, 2])
@pytest.mark.parametrize("G", [2, 3, 4])
@pytest.mark.parametrize("ndm,nchan,nout", [(1, 8, 1), (14, 9, 1016), (16, 67, 1017), (29, 130, 3000), (30, 131, 2032),
                                            (31, 128, 500), (61, 257, 5011)])
def test_block_edges(dpw, G, ndm, nchan, nout, monkeypatch):
    # DM steps that leave a group of few, wide channels few tuples per block (the path needs that)
    _check(monkeypatch, G, dpw, nchan, np.arange(ndm) * min(1.0, nchan / 260.0), nout, ndm)


@pytest.mark.parametrize("dpw", [1, 2])
@pytest.mark.parametrize("G", [2, 3, 4])
@pytest.mark.parametrize("ring", [2, 4])
def test_rings_and_saturation(dpw, G, ring, monkeypatch):
    _check(monkeypatch, G, dpw, 1024, np.arange(33) * 1.0, 1500, 5, full=True, ring=ring)
    _check(monkeypatch, G, dpw, 515, np.arange(47) * 0.5, 1100, 6, ring=ring, band=(1500.0, 1000.0))


@pytest.mark.parametrize("dpw", [1, 2])
def test_unsorted_and_repeated_dms(dpw, monkeypatch):
    dms = np.random.default_rng(3).permutation(np.concatenate([np.arange(40.0), [7.0, 7.0, 0.0, 39.0]]))
    _check(monkeypatch, 3, dpw, 200, dms, 2100, 9)


@pytest.mark.parametrize("dpw", [1, 2])
@pytest.mark.parametrize("G", [2, 4])
def test_several_time_blocks(dpw, G, monkeypatch):
    monkeypatch.setenv("AFGB_PAIR_BUDGET_MB", "24" if G == 2 else "60")
    _check(monkeypatch, G, dpw, 256, np.arange(101) * 2.0, 40 * 1016 + 77, 4)


def test_default_choice_of_block_heights(monkeypatch):
    """Unforced, a wide plan on many tiles and a narrow one on few give the same
    planes as the channel tile kernel."""
    from paper_2511_02328_gb300.search import Plan
    for k in ("AFGB_DEDISP_KERNEL", "AFGB_PAIR_GROUP", "AFGB_PAIR_DPW", "AFGB_PAIR_STAGES"):
        monkeypatch.delenv(k, raising=False)
    for nchan, ndm, nout in ((1024, 301, 60000), (512, 90, 3000)):
        dms = np.arange(ndm) * 1.0
        p = Plan(nchan, 1000.0, 1500.0, 2e-4, dms)
        nsamp = p.dmax + nout
        x = torch.randint(0, 256, (nchan, nsamp), device="cuda", dtype=torch.uint8,
                          generator=torch.Generator(device="cuda").manual_seed(nchan))
        a = p.dedisperse(x)
        monkeypatch.setenv("AFGB_DEDISP_KERNEL", "tile")
        q = Plan(nchan, 1000.0, 1500.0, 2e-4, dms)
        monkeypatch.delenv("AFGB_DEDISP_KERNEL")
        b = q.dedisperse(x)
        assert q.kernel()["path"] == "tile" and torch.equal(a, b)
        p.close()
        q.close()
