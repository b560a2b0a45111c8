"""Fragment scans of many images in one call: exact, and in one go, not one image after another."""
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


@pytest.mark.parametrize("sig", [0, 1, 2])
@pytest.mark.parametrize("n", [2, 4, 5, 40])
@pytest.mark.parametrize("host", [False, True])
def test_uneven_images(cv, sig, n, host):
    """Images of no window, one, some tiles and hundreds, matches at both ends, the tails of each."""
    rng = np.random.default_rng(n)
    file = rng.integers(0, 256, 64 * 20, dtype=np.uint8)
    images = []
    for i in range(n):
        size = int([0, 63, 64, 67, 5000, 40_000, 1_000_003][int(rng.integers(0, 7))] if i else 300_000)
        img = rng.integers(0, 256, size, dtype=np.uint8)
        for at in (0, 128, (size - 64) // 4 * 4, size // 8 * 4):
            if 0 <= at <= size - 64 and rng.random() < 0.7:
                k = int(rng.integers(0, 20))
                img[at:at + 64] = file[64 * k:64 * k + 64]
        images.append(img)
    want = [oracle.frag_match(x, [file, file[:640]]) for x in images]
    devs = images if host else [torch.from_numpy(x).cuda() if x.size else torch.empty(0, dtype=torch.uint8, device="cuda")
                                for x in images]
    torch.cuda.synchronize()
    with cv.master_build([file, file[:640]], signature=sig, unit=cv.CV_UNIT_FRAGMENT) as m:
        for _ in range(2):
            with cv.scan(m, devs) as r:
                for i in range(n):
                    assert np.array_equal(r.matches(i), want[i]), i
                assert r.stats()["sectors"] == sum(max(0, (x.size - 64) // 4 + 1) for x in images)


@pytest.mark.parametrize("sig", [0, 1, 2])
def test_many_images_in_one_go(cv, sig):
    """200 images of 64 KiB take less than ten times what one of them takes, on the device."""
    img = torch.randint(0, 256, (200 << 16,), dtype=torch.uint8, device="cuda")
    images = [img[i << 16:(i + 1) << 16] for i in range(200)]
    file = torch.randint(0, 256, (64 * 5000,), dtype=torch.uint8, device="cuda")
    with cv.master_build([file], signature=sig, unit=cv.CV_UNIT_FRAGMENT) as m:
        t = []
        for xs in (images[:1], images):
            ms = []
            for _ in range(6):
                with cv.scan(m, xs) as r:
                    ms.append(r.stats()["total_ms"])
            t.append(min(ms))
    assert t[1] < 10 * t[0], t
