"""Fragment scans where a tile holds more candidates than usual, and at the edges of its tiles:
repeating data whose every window matches, windows that only share a filter entry, image lengths
around the tile sizes. Bit-exact against the oracle."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

WINDOWS = {0: 32 * 31, 1: 32 * 31, 2: 32 * 23}  # windows per tile, by signature


@pytest.fixture(scope="module")
def cv(cuda_device):
    import __graft_entry__

    __graft_entry__.build()
    from paper_0901_1307_gb300 import cv as cvmod

    return cvmod


def scan(cv, files, img, **kw):
    t = torch.empty(max(img.size, 1), dtype=torch.uint8, device="cuda")
    t[:img.size].copy_(torch.from_numpy(img))
    with cv.master_build(files, unit=cv.CV_UNIT_FRAGMENT, **kw) as m, cv.scan(m, [(t.data_ptr(), img.size)]) as r:
        return r.matches(0)


@pytest.mark.parametrize("sig", [0, 1, 2])
@pytest.mark.parametrize("period", [4, 8, 12, 64, 100])
@pytest.mark.parametrize("bloom", [0, 16])
def test_repeating_data(cv, sig, period, bloom):
    """Every window of a run of repeating data matches (period 4: all with one key; 8 to 64: with
    several; 100: a run of distinct windows), beside fills and random bytes."""
    rng = np.random.default_rng(period)
    unit = rng.integers(0, 256, period, dtype=np.uint8)
    run = np.tile(unit, 30000 // period)
    img = np.concatenate([rng.integers(0, 256, 5000, dtype=np.uint8), run, np.zeros(4000, np.uint8), run[:777],
                          np.full(3001, 255, np.uint8)])
    files = [run[:64 * 9].copy(), rng.integers(0, 256, 640, dtype=np.uint8)]
    want = oracle.frag_match(img, files)
    assert want.size > 1000
    assert np.array_equal(scan(cv, files, img, signature=sig, bloom_bits_per_key=bloom), want)


@pytest.mark.parametrize("sig", [0, 1, 2])
def test_lengths_around_tiles(cv, sig):
    rng = np.random.default_rng(3)
    n = WINDOWS[sig] * 4
    whole = rng.integers(0, 256, 3 * n + 200, dtype=np.uint8)
    files = [whole[n - 256:n + 256].copy(), whole[2 * n:2 * n + 128].copy(), whole[:64].copy()]
    for size in (64, 67, 68, n - 4, n, n + 59, n + 60, n + 63, n + 64, n + 65, 2 * n + 60, 2 * n + 64, 3 * n + 77):
        img = whole[:size].copy()
        img[-64:] = whole[:64]  # the last window matches when the length is a multiple of 4
        assert np.array_equal(scan(cv, files, img, signature=sig), oracle.frag_match(img, files)), size


def test_candidates_that_are_all_rejected(cv):
    """Windows with a master fragment's djb2 and other bytes, one after another: more per lane than
    wait for the filter."""
    rng = np.random.default_rng(4)
    frag = rng.integers(40, 200, 64, dtype=np.uint8)
    col = frag.copy()
    col[10] += 1
    col[11] -= 33
    assert oracle.djb2_64(col) == oracle.djb2_64(frag)
    img = np.concatenate([np.tile(col, 300), frag, np.tile(frag, 40), np.tile(col, 50)])
    assert np.array_equal(scan(cv, [frag], img, signature=2), oracle.frag_match(img, [frag]))


@pytest.mark.parametrize("sig", [0, 1, 2])
@pytest.mark.parametrize("share", [0.02, 0.5, 0.95])
def test_runs_of_equal_words(cv, sig, share):
    """Runs of one word, 1 to 60 words and now and then some tiles long, anywhere: windows that equal the
    one before are not hashed again, and match where that one does."""
    rng = np.random.default_rng(int(100 * share))
    word = np.frombuffer(b"\x11\x22\x33\x44", np.uint32)
    parts, n = [], 0
    while n < 40_000:
        if rng.random() < share:
            k = int(rng.integers(1, 61)) if rng.random() < 0.98 else int(rng.integers(900, 4000))
            parts.append(np.full(k, rng.choice([0, word[0], 0xFFFFFFFF]), np.uint32))
        else:
            parts.append(rng.integers(0, 2**32, int(rng.integers(1, 40)), dtype=np.uint32))
        n += parts[-1].size
    img = np.concatenate(parts).view(np.uint8)
    img = img[:img.size - int(rng.integers(0, 4))]
    files = [np.tile(word, 16).view(np.uint8), img[1000 * 4:1000 * 4 + 640].copy()]
    want = oracle.frag_match(img, files)
    assert want.size > 10
    for bloom in (0, 16):
        assert np.array_equal(scan(cv, files, img, signature=sig, bloom_bits_per_key=bloom), want)


@pytest.mark.parametrize("n_images", [3, 7])
def test_offsets_of_several_images(cv, n_images):
    """Images of none, one and more than 4,096 tiles, the last without any, in one call."""
    rng = np.random.default_rng(n_images)
    frag = rng.integers(0, 256, 128, dtype=np.uint8)
    sizes = [13 << 20, 40, 0, 64, 12_058_624 + 60, 100, 63][-n_images:]
    images = [rng.integers(0, 256, s, dtype=np.uint8) for s in sizes]
    for k, img in enumerate(images):
        for at in (0, 4 * (img.size // 8), img.size // 4 * 4 - 64):
            if 0 <= at <= img.size - 64:
                img[at:at + 64] = frag[64 * (k % 2):][:64]
    devs = [torch.from_numpy(img).cuda() if img.size else torch.empty(16, dtype=torch.uint8, device="cuda") for img in images]
    for sig in (0, 2):
        with cv.master_build([frag], unit=cv.CV_UNIT_FRAGMENT, signature=sig) as m, \
                cv.scan(m, [(d.data_ptr(), img.size) for d, img in zip(devs, images)]) as r:
            for k, img in enumerate(images):
                assert np.array_equal(r.matches(k), oracle.frag_match(img, [frag])), (sig, k)
