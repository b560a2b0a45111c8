"""Lookups in tables without a Bloom filter: tag bytes over the hash layout, against the same masters'
table with a filter (the plain walk over the slots) and the oracle, from tables too small for tags and
windows of tags that wrap around the table's end, up to a table 90% full whose walks are long."""
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


def images_and_files(n, seed):
    rng = np.random.default_rng(seed)
    files = [rng.integers(0, 256, 512 * k, dtype=np.uint8) for k in (n // 2, n - n // 2 - 1, 1) if k]
    files.append(files[0][:512 * 3].copy())  # keys with two postings
    image = rng.integers(0, 256, 512 * (4 * n + 3000), dtype=np.uint8)
    rows = image.reshape(-1, 512)
    src = np.concatenate(files).reshape(-1, 512)
    rows[rng.choice(len(rows), len(src), replace=False)] = src
    return image, files


@pytest.mark.parametrize("sig", [0, 1, 2, 3])
@pytest.mark.parametrize("n", [3, 25, 26, 54, 55, 112, 918, 29_488])  # 25, 54, 112, ...: 32, 64, 128, ... slots, 89% full
@pytest.mark.parametrize("cluster", [0, 1])
def test_tables_without_a_filter(cv, tmp_path, sig, n, cluster):
    image, files = images_and_files(n, 100 * n + sig)
    t = torch.from_numpy(image).cuda()
    kw = dict(signature=sig, position_mode=cluster, max_load=0.9)
    with cv.master_build(files, bloom_bits_per_key=16, **kw) as m, cv.scan(m, [t]) as r:
        want = r.matches(0)
    if not cluster and n < 1000:
        assert np.array_equal(want, oracle.match_hash(image, files))
    for layout in (cv.CV_LAYOUT_HASH, cv.CV_LAYOUT_SORTED, cv.CV_LAYOUT_AUTO):
        with cv.master_build(files, bloom_bits_per_key=0, layout=layout, **kw) as m:
            path = str(tmp_path / "t")
            cv.master_save(m, path)
            with cv.master_load(path) as again:
                assert again.info() == m.info()
                for table in (m, again):
                    with cv.scan(table, [t]) as r:
                        assert np.array_equal(r.matches(0), want)
            with cv.batch_create(m, [t]) as b:
                b.run()
                assert np.array_equal(cv.device_matches_to_numpy(b.matches(0)), want)


@pytest.mark.parametrize("sig", [2, 3])
def test_sorted_keys_in_one_bucket(cv, sig):
    """Signatures whose low words (the sorted keys) are nearly all in one bucket of the index: sectors of
    zeros but for their last bytes."""
    rng = np.random.default_rng(sig)
    rows = np.zeros((9000, 512), np.uint8)
    rows[:, 510:] = rng.permutation(65536)[:9000].astype(">u2").view(np.uint8).reshape(-1, 2)
    image = np.concatenate([rows[::2], rng.integers(0, 256, (500, 512), dtype=np.uint8), rows[:7000:3]]).reshape(-1)
    files = [rows[:4000].reshape(-1), rows[4000:6500].reshape(-1)]
    t = torch.from_numpy(image).cuda()
    with cv.master_build(files, signature=sig, layout=cv.CV_LAYOUT_SORTED, bloom_bits_per_key=0) as m:
        with cv.scan(m, [t]) as r:
            assert np.array_equal(r.matches(0), oracle.match_hash(image, files))
