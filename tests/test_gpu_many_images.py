"""As many images in a call as its counts fill the pinned staging, one more and one less: counts beyond it
are read into pageable memory. Sector and fragment scans, results on the host and on the device."""
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


# 512 counts are staged; a sector scan has four more of them than images, a fragment scan three
@pytest.mark.parametrize("n", [507, 508, 509, 510, 512, 513, 1100])
@pytest.mark.parametrize("unit", [0, 1])
def test_counts_around_the_stage(cv, n, unit):
    rng = np.random.default_rng(n)
    size = 64 if unit else 512
    file = rng.integers(0, 256, size * 6, dtype=np.uint8)
    images = []
    for i in range(n):
        img = rng.integers(0, 256, size * int(rng.integers(1, 9)) + int(rng.integers(0, 60)), dtype=np.uint8)
        if i % 5 == 0 or i == n - 1:
            img[:size] = file[size * (i % 6):][:size]
        images.append(img if i % 97 else img[:size // 2])  # some without a sector or window
    want = [oracle.frag_match(x, [file]) if unit else oracle.match_hash(x, [file]) for x in images]
    assert sum(w.size for w in want) > 90 and want[-1].size
    devs = [torch.from_numpy(x).cuda() for x in images]
    torch.cuda.synchronize()
    for sig in (0, 2):
        with cv.master_build([file], unit=unit, signature=sig) as m:
            for keep in (False, True):
                with cv.scan(m, devs, keep_on_device=keep) as r:
                    for i in range(n):
                        got = cv.device_matches_to_numpy(r.matches(i)) if keep else r.matches(i)
                        assert np.array_equal(got, want[i]), (sig, keep, i)
