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
