"""Group-row reservations on a device without room for the fastest set's rows:
shorter time blocks where some memory is left, the channel tile kernel where
hardly any is, the same plane either way, and the full reservation again once the
memory is back."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BAND, TSAMP = (1000.0, 1500.0), 2e-4


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _plane(p, x):
    from paper_2511_02328_gb300 import _lib
    nout = p.nout(x.shape[1])
    plane = torch.empty((p.ndm, nout), dtype=torch.int32, device="cuda")
    _lib.af_dedisperse(p.handle, x.data_ptr(), x.shape[1], plane.data_ptr(), 0, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return plane


@pytest.mark.parametrize("dpw", [0, 2])  # every set, or none of 15-row blocks
@pytest.mark.parametrize("left_mb,path", [(400, "pairs"), (48, "tile")])
def test_reserve_with_little_memory_left(dpw, left_mb, path, monkeypatch):
    from paper_2511_02328_gb300 import _lib
    from paper_2511_02328_gb300.search import Plan
    for k in ("AFGB_DEDISP_KERNEL", "AFGB_PAIR_GROUP", "AFGB_PAIR_DPW", "AFGB_PAIR_STAGES", "AFGB_PAIR_BUDGET_MB"):
        monkeypatch.delenv(k, raising=False)
    if dpw:
        monkeypatch.setenv("AFGB_PAIR_DPW", str(dpw))
    nchan, nout, dms = 1024, 60000, np.arange(0.0, 301.0, 1.0)
    p, q = Plan(nchan, *BAND, TSAMP, dms), Plan(nchan, *BAND, TSAMP, dms)
    nsamp = p.dmax + nout
    x = torch.randint(0, 256, (nchan, nsamp), device="cuda", dtype=torch.uint8,
                      generator=torch.Generator(device="cuda").manual_seed(left_mb))
    ref = _plane(q, x)  # nothing reserved: the channel tile kernel
    assert q.kernel()["path"] == "tile"
    assert _lib.af_dedisperse_workspace_size(p.handle, nsamp) > left_mb << 20
    q.reserve(nsamp)
    assert q.kernel()["path"] == "pairs" and torch.equal(_plane(q, x), ref)  # with room; the kernels are loaded
    q.close()
    spare = torch.empty_like(ref)
    del spare  # the plane below comes from torch's own pool
    free = torch.cuda.mem_get_info()[0]
    fill = torch.empty(free - (left_mb << 20), dtype=torch.uint8, device="cuda")
    try:
        _lib.af_dedisperse_reserve(p.handle, nsamp)
        assert p.kernel()["path"] == path
        if path == "pairs":
            _lib.af_dedisperse_timing(p.handle, 1)
        assert torch.equal(_plane(p, x), ref)
        if path == "pairs":  # several blocks of a buffer within what was left
            assert _lib.af_dedisperse_times(p.handle, 0)[2] > left_mb << 20
            _lib.af_dedisperse_timing(p.handle, 0)
    finally:
        del fill
        torch.cuda.empty_cache()
    _lib.af_dedisperse_reserve(p.handle, nsamp)
    assert p.kernel()["path"] == "pairs" and torch.equal(_plane(p, x), ref)
    p.close()
