"""Logits into any buffer of the caller's: at any byte address, and over the images
themselves (written once every image has been read)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("n", [1, 7, 40, 153, 260])
def test_logits_buffers(n):
    from paper_2511_02328_gb300 import _lib
    m = _lib.af_model_create(512, 3)
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.rand((n, 64, 64, 2), generator=g, device="cuda").to(torch.bfloat16)
    ref = torch.empty((n, 2), device="cuda")
    _lib.af_model_forward(m, x.data_ptr(), n, ref.data_ptr(), 0)
    want = ref.cpu().numpy()
    assert np.isfinite(want).all() and np.ptp(want) > 0
    for offset in (1, 2, 4, 6):
        buf = torch.zeros(8 * n + 16, dtype=torch.uint8, device="cuda")
        _lib.af_model_forward(m, x.data_ptr(), n, buf.data_ptr() + offset, 0)
        got = buf.cpu().numpy()
        assert np.array_equal(got[offset:offset + 8 * n].view(np.float32).reshape(n, 2), want)
        assert not got[:offset].any() and not got[offset + 8 * n:].any()
    # over the images: all 8 n bytes of the first image's, and the last 8 n of the buffer's
    for at in (0, x.numel() * 2 - 8 * n):
        y = x.clone()
        _lib.af_model_forward(m, y.data_ptr(), n, y.data_ptr() + at, 0)
        raw = y.view(torch.uint8).reshape(-1)[at:at + 8 * n].cpu().numpy()
        assert np.array_equal(raw.view(np.float32).reshape(n, 2), want)
    _lib.af_model_destroy(m)
