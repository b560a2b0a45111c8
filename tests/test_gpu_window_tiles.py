"""cv_window_signatures at the edges of its tiles (32 lanes of 17 djb2 or 31 MD5 windows) and beyond the
grid's first round, against the oracle."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cv(cuda_device):
    import __graft_entry__

    __graft_entry__.build()
    from paper_0901_1307_gb300 import cv as cvmod

    return cvmod


@pytest.mark.parametrize("sig,win", [(0, 992), (1, 992), (2, 544)])
@pytest.mark.parametrize("tiles", [1, 2, 8, 9])
@pytest.mark.parametrize("more", [-4, 0, 1, 4, 67])
def test_lengths_around_tiles(cv, sig, win, tiles, more):
    n = 4 * win * tiles + 60 + more  # 4 win tiles + 60 bytes hold whole tiles of windows
    img = np.random.default_rng(n).integers(0, 256, n, dtype=np.uint8)
    count = (n - 64) // 4 + 1
    d = torch.from_numpy(img).cuda()
    out = torch.full((count + 1, 16), 0xA5, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    cv.window_signatures(d.data_ptr(), n, sig, out.data_ptr())
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    width = 8 if sig == 2 else 16
    assert np.array_equal(got[:count, :width], oracle.window_signatures(img, sig)[:, :width])
    assert (got[count] == 0xA5).all()
