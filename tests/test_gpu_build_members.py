"""Keys with several members among keys with one: every duplicate is reported, in file order, for
tables built from master sets in which none, some, most or all sectors repeat, with the copies in
one file, in many, and on both sides of a chunk of slots."""
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


def masters(rng, n, distinct, files):
    """n sectors drawn from `distinct` random ones (some all equal: left out), cut into files."""
    pool = rng.integers(0, 256, (distinct, 512), dtype=np.uint8)
    pool[rng.integers(0, distinct, distinct // 10)] = 7
    rows = pool[rng.integers(0, distinct, n)] if distinct < n else pool[:n]
    cuts = np.sort(rng.integers(0, n + 1, files - 1))
    return pool, [np.ascontiguousarray(x).ravel() for x in np.split(rows, cuts)]


# sectors, distinct ones, files: no key with several; pairs; a few; one key with all; many of many
@pytest.mark.parametrize("n,distinct,files", [(5000, 5000, 40), (3000, 2000, 30), (2048, 300, 1), (1500, 1, 9),
                                              (40000, 37, 500), (1, 1, 1)])
@pytest.mark.parametrize("sig", [0, 3])
def test_members_in_master_order(cv, n, distinct, files, sig):
    rng = np.random.default_rng(n + distinct)
    pool, parts = masters(rng, n, distinct, files)
    img = np.concatenate([pool[rng.integers(0, distinct, 20)].ravel(), rng.integers(0, 256, 5120, dtype=np.uint8)])
    want = oracle.match_hash(img, parts)
    t = torch.from_numpy(img).cuda()
    for kw in ({}, {"layout": cv.CV_LAYOUT_SORTED}, {"position_mode": cv.CV_POSITION_CLUSTER, "max_load": 0.9}):
        with cv.master_build(parts, signature=sig, **kw) as m, cv.scan(m, [t]) as r:
            ref = oracle.match_position(img, parts, 0) if "position_mode" in kw else want
            assert np.array_equal(r.matches(0), ref), kw
            kept = sum(int((p.reshape(-1, 512) != p.reshape(-1, 512)[:, :1]).any(axis=1).sum()) for p in parts if p.size)
            assert m.info()["n_kept"] == kept


def test_members_of_fragments(cv):
    rng = np.random.default_rng(5)
    pool = rng.integers(0, 256, (50, 64), dtype=np.uint8)
    parts = [np.ascontiguousarray(pool[rng.integers(0, 50, k)]).ravel() for k in rng.integers(1, 200, 30)]
    img = np.concatenate([parts[3], parts[7][:1000], rng.integers(0, 256, 4000, dtype=np.uint8)])
    want = oracle.frag_match(img, parts)
    t = torch.from_numpy(img).cuda()
    for sig in (0, 2):
        with cv.master_build(parts, signature=sig, unit=cv.CV_UNIT_FRAGMENT) as m, cv.scan(m, [t]) as r:
            assert np.array_equal(r.matches(0), want)


@pytest.mark.parametrize("n", [(1 << 18) - 1, 1 << 18, (1 << 18) + 767, 393_217])
@pytest.mark.parametrize("copies", [0, 1, 1000])
def test_inserts_of_many_keys(cv, n, copies):
    """Around the number of keys from which the insert takes them by chunks of 768: sectors told apart by
    their first bytes, runs of copies among them (within a warp and across), and fills left out."""
    rng = np.random.default_rng(n)
    ids = np.arange(n, dtype=np.uint32)
    for at in rng.integers(0, n - 1100, 8 if copies else 0):
        ids[at:at + copies + 1] = ids[at]
    rows = np.zeros((n, 512), np.uint8)
    rows[:, :4] = (ids[:, None] >> np.array([0, 8, 16, 24], np.uint32)).astype(np.uint8)
    rows[:, 4] = 1
    rows[5000] = 0
    dev = torch.from_numpy(rows).cuda()
    with cv.master_build([dev.view(-1)]) as m, cv.scan(m, [dev.view(-1)]) as r:
        info, got = m.info(), r.matches(0)
    live = np.delete(ids, 5000)
    _, inverse, counts = np.unique(live, return_inverse=True, return_counts=True)
    assert info["n_kept"] == n - 1 and info["n_unique"] == counts.size
    assert got.size == int(counts[inverse].sum())
    # every sector finds itself, and each match is of the sector's own bytes, in order
    assert np.array_equal(ids[got["disk_sector"]], ids[got["file_sector"]])
    assert (got["disk_sector"] == got["file_sector"]).sum() == n - 1
    assert np.array_equal(np.lexsort((got["file_sector"], got["disk_sector"])), np.arange(got.size))
