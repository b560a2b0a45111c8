"""The second half of a scan, offsets and expansion in one launch over groups of 512 output tiles of 32
sectors: sizes around a chunk, many groups and the end of the last one, many postings per key, more
matches than there is room for at first, images without matches, several images, and results that a
first scan sized wrongly."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CHUNK = 512 * 32  # sectors of a group


@pytest.fixture(scope="module")
def cv(cuda_device):
    import __graft_entry__

    __graft_entry__.build()
    from paper_0901_1307_gb300 import cv as cvmod

    return cvmod


@pytest.mark.parametrize("n", [1, 31, 33, 128 * 32 + 5, CHUNK - 1, CHUNK, CHUNK + 1, 256 * CHUNK - 128, 256 * CHUNK + 1])
def test_sizes_around_a_group(cv, n):
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


@pytest.mark.parametrize("nosec", [4096 * 512 * 32 + 100])
def test_groups_of_more_than_one_chunk(cv, nosec):
    """Above 2^21 output tiles a group is 1,024 tiles: an offset follows from the chunk before it."""
    if torch.cuda.mem_get_info()[0] < nosec * 600:
        pytest.skip("not enough device memory")
    img = torch.zeros(nosec * 512, dtype=torch.uint8, device="cuda")
    at = sorted({*range(0, nosec, 99_991), *range(1024 * 32 * 7 - 40, 1024 * 32 * 7 + 40), nosec - 1})
    rows = torch.randint(1, 256, (len(at), 512), dtype=torch.uint8, device="cuda",
                         generator=torch.Generator("cuda").manual_seed(3))
    img.view(nosec, 512)[torch.tensor(at, device="cuda")] = rows
    cut = 64 << 20  # several images of one allocation: segments begin within groups
    parts = [img[:512 * 1000], img[512 * 1000:512 * cut + 512 * 77], img[512 * cut + 512 * 77:]]
    with cv.master_build([rows.reshape(-1)]) as m:
        with cv.scan(m, [img]) as r:
            got = r.matches(0)
            assert got["disk_sector"].tolist() == at and got["file_sector"].tolist() == list(range(len(at)))
        with cv.scan(m, parts) as r:
            first, k = 0, 0
            for i, p in enumerate(parts):
                n = p.numel() // 512
                want = [a - first for a in at if first <= a < first + n]
                got = r.matches(i)
                assert got["disk_sector"].tolist() == want
                assert got["file_sector"].tolist() == list(range(k, k + len(want)))
                first, k = first + n, k + len(want)
