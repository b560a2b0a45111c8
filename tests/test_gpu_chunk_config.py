"""The scan configuration follows what one launch scans: the device images together, or one chunk of a
host image, however long the image."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MIB = 1 << 20


@pytest.fixture(scope="module")
def cv(cuda_device):
    import __graft_entry__

    __graft_entry__.build()
    from paper_0901_1307_gb300 import cv as cvmod

    return cvmod


@pytest.mark.parametrize("sig,mib,chunk_mib", [(0, 128, 1), (0, 128, 64), (0, 64, 0), (0, 128, 128), (0, 300, 0),
                                               (1, 1024, 16), (1, 1024, 0), (1, 1024, 1024), (2, 128, 1), (3, 32, 1)])
def test_host_images(cv, sig, mib, chunk_mib):
    img = torch.zeros(mib * MIB, dtype=torch.uint8)
    rng = np.random.default_rng(mib)
    file = rng.integers(0, 256, 512 * 9, dtype=np.uint8)
    img[512 * 77:512 * 86] = torch.from_numpy(file)
    img[-512 * 9:] = torch.from_numpy(file)
    launch = mib if sig > 1 else min(mib, chunk_mib or 256)
    with cv.master_build([file], signature=sig) as m:
        with cv.scan(m, [img[:launch * MIB].cuda()]) as r:  # a device image of one launch's length
            want = r.stats()["kernel_config"]
        with cv.scan(m, [img], chunk_bytes=chunk_mib * MIB) as r:
            assert cv.kernel_configs()[r.stats()["kernel_config"]] == cv.kernel_configs()[want]
            got = r.matches(0)
    at = np.concatenate([np.arange(77, 86), np.arange(9) + mib * 2048 - 9])
    assert np.array_equal(got["disk_sector"], at) and np.array_equal(got["file_sector"], np.tile(np.arange(9), 2))


def test_host_and_device_images(cv):
    """Device images count together, a host image by its chunk; the larger of the two decides."""
    rng = np.random.default_rng(1)
    file = rng.integers(0, 256, 512 * 9, dtype=np.uint8)
    host = torch.zeros(100 * MIB, dtype=torch.uint8)
    host[:file.size] = torch.from_numpy(file)
    dev = host.cuda()
    with cv.master_build([file]) as m:
        def config(images, chunk):
            with cv.scan(m, images, chunk_bytes=chunk) as r:
                for i in range(len(images)):
                    assert np.array_equal(r.matches(i), oracle.match_hash(file, [file]))
                return r.stats()["kernel_config"]
        small, large = config([dev[:MIB]], 0), config([dev], 0)
        assert small != large
        assert config([host, dev[:MIB]], MIB) == small
        assert config([host, dev[:60 * MIB], dev[:60 * MIB]], MIB) == large
        assert config([dev[:MIB], host], 0) == large
