"""Tiles handed out while the scan runs: every sector is hashed exactly once, whether an image is
part of one tile, one tile, a few, or many times what the GPU holds at once."""
import numpy as np
import pytest

import oracle
from paper_0901_1307_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cv(cuda_device):
    import __graft_entry__

    __graft_entry__.build()
    from paper_0901_1307_gb300 import cv as cvmod

    return cvmod


# one sector; around a 256-sector tile; 152 SMs x 4 blocks of one tile each, and one sector more;
# several rounds of that with a ragged last tile
@pytest.mark.parametrize("n", [1, 255, 256, 257, 608 * 256, 608 * 256 + 1, 300001])
def test_every_sector_hashed_once(cv, n):
    img = synth.random_sectors(n, n)
    dev = torch.from_numpy(img).cuda()
    out = torch.zeros(n * 16, dtype=torch.uint8, device="cuda")
    cv.sector_signatures(dev.data_ptr(), n, cv.CV_SIG_MD5, out.data_ptr())
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy().reshape(n, 16), oracle.md5_sectors(img))


@pytest.mark.parametrize("cfg", range(9))
def test_many_tiles_every_configuration(cv, cfg):
    """Two images whose tiles outnumber the resident blocks of every configuration (at most 152 x
    32), each ending inside a tile, with matches in the first and the last sector."""
    n = 152 * 32 * 64 + 77
    img = torch.randint(0, 256, (n * 512,), dtype=torch.uint8, device="cuda",
                        generator=torch.Generator("cuda").manual_seed(cfg))
    file = torch.cat([img[:512], img[-512:]])
    with cv.master_build([file]) as m, cv.scan(m, [img, img[: 512 * 1001]], kernel_config=cfg + 1) as r:
        got = [tuple(int(x) for x in row) for row in r.matches(0)]
        assert got == [(0, 0, 0), (n - 1, 0, 1)]
        assert [tuple(int(x) for x in row) for row in r.matches(1)] == [(0, 0, 0)]
