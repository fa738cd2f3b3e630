"""A reservation holds for every input up to its length: a later, shorter one
neither changes the row set picked for the longer one nor shortens its time
blocks, and a call shorter than the reservation writes only its own tiles' rows."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BAND, TSAMP = (1000.0, 1500.0), 2e-4


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _call(p, x):
    """(plane, row bytes written, window bytes copied) of one dedispersion by the C call alone."""
    from paper_2511_02328_gb300 import _lib
    _lib.af_dedisperse_timing(p.handle, 1)
    nout = p.nout(x.shape[1])
    plane = torch.empty((p.ndm, nout), dtype=torch.int32, device="cuda")
    _lib.af_dedisperse(p.handle, x.data_ptr(), x.shape[1], plane.data_ptr(), 0, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return plane, _lib.af_dedisperse_times(p.handle, 0)[2:]


# lengths whose picks differ: other group sizes, other block heights
@pytest.mark.parametrize("nchan,ndm,long,short", [(512, 609, 20000, 2000), (256, 301, 20000, 8000), (1024, 301, 8000, 2000)])
@pytest.mark.parametrize("search", [False, True])
def test_shorter_reservation_keeps_the_longer(nchan, ndm, long, short, search, monkeypatch):
    from paper_2511_02328_gb300 import _lib
    from paper_2511_02328_gb300.search import Plan
    for k in ("AFGB_PAIR_GROUP", "AFGB_PAIR_DPW", "AFGB_PAIR_STAGES", "AFGB_PAIR_BUDGET_MB"):
        monkeypatch.delenv(k, raising=False)
    monkeypatch.setenv("AFGB_DEDISP_KERNEL", "pairs")  # rows even where channel tiles are faster
    dms = np.arange(ndm) * 1.0
    own = Plan(nchan, *BAND, TSAMP, dms)  # what the short length would pick by itself
    own.reserve(own.dmax + short)
    p = Plan(nchan, *BAND, TSAMP, dms)
    n = p.dmax + long
    x = torch.randint(0, 256, (nchan, n), device="cuda", dtype=torch.uint8,
                      generator=torch.Generator(device="cuda").manual_seed(nchan + ndm))
    if search:
        _lib.af_search_reserve(p.handle, n, 4096)
    else:
        _lib.af_dedisperse_reserve(p.handle, n)
    before = p.kernel()
    assert before["path"] == own.kernel()["path"] == "pairs" and before != own.kernel()
    full, moved = _call(p, x)
    xs = x[:, :p.dmax + short].contiguous()
    _lib.af_dedisperse_reserve(p.handle, xs.shape[1])
    assert p.kernel() == before
    again, moved_again = _call(p, x)
    assert torch.equal(again, full) and moved_again == moved
    part, moved_part = _call(p, xs)
    assert torch.equal(part, full[:, :short]) and moved_part[0] < moved[0]
    if search:
        h = x.cpu().numpy()
        _, total = _lib.af_search(p.handle, h, n, [1, 4, 16], 6.0, 4096)
        q = Plan(nchan, *BAND, TSAMP, dms)
        _, ref = q.search_host(h, [1, 4, 16], 6.0, cap=4096)
        assert total == ref
        q.close()
    p.close()
    own.close()
