"""Tables of many sectors that are copies of few, in the order in which they queue at the fewest slots:
every copy is found, in master order, and the build does not wait for them one by one."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cv(cuda_device):
    import __graft_entry__

    __graft_entry__.build()
    from paper_0901_1307_gb300 import cv as cvmod

    return cvmod


def sectors(ids):
    """Sectors that begin with their id, not all bytes equal."""
    rows = torch.zeros((ids.numel(), 512), dtype=torch.uint8, device="cuda")
    for k in range(4):
        rows[:, k] = (ids >> (8 * k)) & 255
    rows[:, 4] = 1
    return rows.view(-1)


@pytest.mark.parametrize("kw", [{}, {"bloom_bits_per_key": 0, "max_load": 0.9}, {"signature": 3}])
@pytest.mark.parametrize("pattern", ["equal", "two", "three", "pairs", "37 drawn", "some"])
def test_copies_in_master_order(cv, pattern, kw):
    n = (1 << 18) + 1000
    i = torch.arange(n, device="cuda")
    g = torch.Generator("cuda").manual_seed(1)
    ids = {"equal": i * 0, "two": i % 2, "three": i % 3, "pairs": (i // 2) % 5,
           "37 drawn": torch.randint(0, 37, (n,), generator=g, device="cuda"),
           "some": torch.where(torch.rand(n, generator=g, device="cuda") < 0.01, i % 7, i)}[pattern]
    table = sectors(ids)
    probe = torch.unique(ids)[:40]
    with cv.master_build([table], **kw) as m, cv.scan(m, [sectors(probe)], keep_on_device=True) as r:
        info = m.info()
        got = torch.as_tensor(r.matches(0), device="cuda").view(torch.int64).clone()
    assert info["n_kept"] == n and info["n_unique"] == torch.unique(ids).numel()
    want = torch.cat([torch.nonzero(ids == p)[:, 0] for p in probe])
    assert torch.equal(got[:, 1] >> 32, want)
    count = torch.stack([(ids == p).sum() for p in probe])
    assert torch.equal(got[:, 0], torch.arange(probe.numel(), device="cuda").repeat_interleave(count))


def test_equal_sectors_do_not_queue(cv):
    """A table of 2^20 equal sectors is built in at most two and a half times the time of one of 2^20
    different ones."""
    i = torch.arange(1 << 20, device="cuda")
    best = []
    for ids in (i, i * 0):
        table = sectors(ids)
        torch.cuda.synchronize()
        t = []
        for _ in range(8):
            a = time.perf_counter()
            cv.master_build([table]).close()
            t.append(time.perf_counter() - a)
        best.append(min(t))
    assert best[1] < 2.5 * best[0], best


def test_large_tables_are_not_paid_for_twice(cv):
    """A table with an array of more than 1 GiB (the sectors' copies of a 64-bit signature) is built and freed
    in less than four and a half times what one of half the sectors takes, which fits what is kept."""
    best = []
    for n in (1_500_000, 3_000_000):
        table = torch.randint(-2**31, 2**31 - 1, (n * 128,), dtype=torch.int32, device="cuda").view(torch.uint8)
        t = []
        for _ in range(8):
            torch.cuda.synchronize()
            a = time.perf_counter()
            m = cv.master_build([table], signature=2)
            info = m.info()
            m.close()
            t.append(time.perf_counter() - a)
        best.append(min(t))
        assert info["n_unique"] == n
    assert best[1] < 4.5 * best[0], best
