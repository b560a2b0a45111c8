"""The second half of a scan in one launch and in three: sizes around the limit between them, many
postings per key, more matches than there is room for at first, images without matches, several
images, and results that a first scan sized wrongly."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LIMIT = (1 << 17) * 32  # sectors: output tiles of the one-launch form, 32 sectors each


@pytest.fixture(scope="module")
def cv(cuda_device):
    import __graft_entry__

    __graft_entry__.build()
    from paper_0901_1307_gb300 import cv as cvmod

    return cvmod


@pytest.mark.parametrize("n", [1, 31, 33, 128 * 32 + 5, LIMIT - 128, LIMIT, LIMIT + 1])
def test_sizes_around_the_limit(cv, n):
    """Matches in the first and last sector and every 4,097th between."""
    img = torch.randint(0, 256, (n * 512,), dtype=torch.uint8, device="cuda",
                        generator=torch.Generator("cuda").manual_seed(n))
    at = sorted({0, n - 1, *range(0, n, 4097)})
    rows = img.view(n, 512)[torch.tensor(at, device="cuda")].contiguous()
    with cv.master_build([rows.reshape(-1)]) as m:
        for _ in range(2):  # the second scan has the first one's count to go by
            with cv.scan(m, [img]) as r:
                got = r.matches(0)
                assert got["disk_sector"].tolist() == at and got["file_sector"].tolist() == list(range(len(at)))
                assert r.stats()["hit_sectors"] == len(at)


@pytest.mark.parametrize("sig", [0, 2])
def test_many_postings_and_images(cv, sig):
    """A sector with 3,000 copies in the master files, in images with and without it; the counts of
    one scan are no guide to the next one's."""
    rng = np.random.default_rng(sig)
    common = rng.integers(0, 256, 512, dtype=np.uint8)
    files = [np.tile(common, 100) for _ in range(30)] + [rng.integers(0, 256, 5120, dtype=np.uint8)]
    none = rng.integers(0, 256, 512 * 700, dtype=np.uint8)
    some = none.copy()
    for s in (0, 5, 31, 32, 64, 699):
        some[512 * s:512 * s + 512] = common
    some[512 * 40:512 * 50] = files[-1]
    images = [none, some, none[:511], some[:512 * 33], none, some, none]
    with cv.master_build(files, signature=sig) as m:
        for pick in ([1], [0], list(range(7)), [1, 3], [4], [1, 1, 1, 1, 1]):
            devs = [torch.from_numpy(images[k]).cuda() for k in pick]
            for keep in (False, True):
                with cv.scan(m, devs, keep_on_device=keep) as r:
                    for i, k in enumerate(pick):
                        got = cv.device_matches_to_numpy(r.matches(i)) if keep else r.matches(i)
                        assert np.array_equal(got, oracle.match_hash(images[k], files)), (pick, i)


def test_rejected_and_kept_postings_of_one_key(cv):
    """A 64-bit signature's key whose postings partly differ from the disk sector."""
    rng = np.random.default_rng(9)
    a = rng.integers(40, 200, 512, dtype=np.uint8)
    b = a.copy()
    b[100] += 1
    b[101] -= 33
    assert oracle.djb2_64(a) == oracle.djb2_64(b)
    files = [np.concatenate([a, b, a]), np.concatenate([b, b]), a]
    img = np.concatenate([a, b, rng.integers(0, 256, 512, dtype=np.uint8), b, a])
    t = torch.from_numpy(img).cuda()
    with cv.master_build(files, signature=2) as m, cv.scan(m, [t]) as r:
        assert np.array_equal(r.matches(0), oracle.match_hash(img, files))
        assert r.stats()["confirm_rejected"] == 2 * 3 + 2 * 3
