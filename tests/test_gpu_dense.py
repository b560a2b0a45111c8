"""Images most of whose sectors match, with one master copy or many: the offsets and expansion of groups
of 32 to 512 output tiles of 32 sectors, spread over the GPU."""
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


def rows(cv, r, i=0):
    """(disk sector, file, file sector) of image i as int64[n, 3]."""
    m = r.matches(i)
    t = torch.as_tensor(m, device="cuda").view(torch.int64) if m.n else torch.empty((0, 2), dtype=torch.int64, device="cuda")
    return torch.stack([t[:, 0], t[:, 1] & 0xFFFFFFFF, t[:, 1] >> 32], dim=1)


# sectors: one tile, the edges of a group of 32, 64, 128, 256 and 512 tiles, the sizes where groups grow
@pytest.mark.parametrize("n", [1, 1023, 1025, 304 * 1024, 304 * 1024 + 1, 608 * 1024 - 31, 608 * 1024 + 33,
                               1216 * 1024 + 1, 4864 * 1024 + 1])
@pytest.mark.parametrize("sig", [0, 3])
def test_every_sector_matches(cv, n, sig):
    """All sectors but two match a sector of which one, two and three copies are in three files."""
    g = torch.Generator("cuda").manual_seed(n)
    key = torch.randint(0, 256, (3, 512), generator=g, dtype=torch.uint8, device="cuda")
    files = [key.reshape(-1), key[1:].reshape(-1).contiguous(), key[2:].reshape(-1).contiguous()]
    which = torch.arange(n, device="cuda") % 3
    img = key[which]
    out = [n // 2, n - 1] if n > 2 else []
    for at in out:
        img[at] = 0
    keep = torch.ones(n, dtype=torch.bool, device="cuda")
    keep[out] = False
    s, w = torch.arange(n, device="cuda")[keep], which[keep]
    s = s.repeat_interleave(w + 1)
    first = torch.cumsum(w + 1, 0) - (w + 1)
    f = torch.arange(s.numel(), device="cuda") - first.repeat_interleave(w + 1)
    want = torch.stack([s, f, w.repeat_interleave(w + 1) - f], dim=1)
    with cv.master_build(files, signature=sig) as m:
        for _ in range(2):
            with cv.scan(m, [img.view(-1)], keep_on_device=True) as r:
                assert r.stats()["hit_sectors"] == int(keep.sum())
                assert torch.equal(rows(cv, r), want)


def test_many_copies_are_written_by_the_whole_gpu(cv):
    """32 MiB of one sector with 128 master copies: 134 MB of matches in less than a millisecond."""
    key = torch.randint(0, 256, (512,), dtype=torch.uint8, device="cuda")
    img, file = key.repeat(1 << 16), key.repeat(128)
    ms = []
    with cv.master_build([file]) as m:
        for _ in range(5):
            with cv.scan(m, [img], keep_on_device=True) as r:
                st = r.stats()
                assert st["matches"] == 1 << 23
                ms.append(st["total_ms"] - st["kernel_ms"])
    assert min(ms) < 1.0, ms


@pytest.mark.parametrize("cap", [0, 1, 77, 4095, 4096, 5000])
def test_too_little_room(cv, cap):
    """A batch with room for cap of 4,096 matches: those images whose matches fit are right, the count is."""
    key = torch.randint(0, 256, (512,), dtype=torch.uint8, device="cuda")
    images = [key.repeat(8) for _ in range(4)]
    with cv.master_build([key.repeat(128)]) as m, cv.batch_create(m, images, match_capacity=cap or 4096 + 1) as b:
        b.run()
        if cap and cap < 4096:
            with pytest.raises(cv.CVError) as e:
                b.wait()
            assert e.value.code == cv.CV_ERANGE
        else:
            assert b.wait() == 4096
        for i in range(4):
            if 1024 * (i + 1) > (cap or 4097):
                with pytest.raises(cv.CVError):
                    b.matches(i)
                continue
            got = cv.device_matches_to_numpy(b.matches(i))
            assert np.array_equal(got["disk_sector"], np.repeat(np.arange(8), 128))
            assert np.array_equal(got["file_sector"], np.tile(np.arange(128), 8))
