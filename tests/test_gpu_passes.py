"""The passes after a scan, driven with the scratch that a caller of the C ABI has no say over (passes.cu):
passes without room for every match."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
PACKAGE = os.path.join(os.path.dirname(HERE), "paper_0901_1307_gb300")
ST_OVERFLOW = 8


@pytest.fixture(scope="module")
def cv(cuda_device):
    import __graft_entry__

    __graft_entry__.build()
    from paper_0901_1307_gb300 import cv as cvmod

    return cvmod


@pytest.fixture(scope="module")
def passes(cv, tmp_path_factory):
    from paper_0901_1307_gb300 import build

    lib = str(tmp_path_factory.mktemp("passes") / "passes.so")
    cv.load()
    subprocess.run([build._nvcc(), "-shared", "-cudart", "shared", *build.ARCH, *build.FLAGS,
                    os.path.join(HERE, "passes.cu"), "-o", lib, "-L" + PACKAGE, "-lcv", "-Xlinker", "-rpath",
                    "-Xlinker", PACKAGE], check=True)
    return ctypes.CDLL(lib)


def scan(passes, m, img, n, cap, all_or_none, room):
    """(total, status, sectors with a match, output as int64[room, 2], -1 where nothing was written)."""
    out = torch.full((room, 2), -1, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    h = (ctypes.c_uint64 * 3)()
    u64, vp = ctypes.c_uint64, ctypes.c_void_p
    rc = passes.passes_scan(vp(m.handle), vp(img.data_ptr()), u64(n), u64(cap), ctypes.c_int(all_or_none),
                            vp(out.data_ptr()), h)
    assert rc == 0
    return int(h[0]), int(h[1]) & 0xFFFFFFFF, int(h[2]), out


@pytest.mark.parametrize("sig", [0, 2])
@pytest.mark.parametrize("n", [40, 5000, 400_000])
def test_room_for_all_or_none(cv, passes, sig, n):
    """Without room for every match, one short or none at all, the pass writes nothing, says so, and has
    counted; with room it writes all; where a part is wanted, that part."""
    g = torch.Generator("cuda").manual_seed(n)
    key = torch.randint(0, 256, (2, 512), generator=g, dtype=torch.uint8, device="cuda")
    which = torch.arange(n, device="cuda") % 3
    img = torch.where((which < 2)[:, None], key[which.clamp(max=1)], torch.zeros(512, dtype=torch.uint8, device="cuda"))
    hits = int((which < 2).sum())
    total = 3 * int((which == 0).sum()) + int((which == 1).sum())
    with cv.master_build([key[0].repeat(3), key[1]], signature=sig) as m:
        with cv.scan(m, [img.view(-1)], keep_on_device=True) as r:
            want = torch.as_tensor(r.matches(0), device="cuda").view(torch.int64).clone()
        assert want.shape[0] == total
        for cap in (0, 1, total - 1):
            t, status, h, out = scan(passes, m, img, n, cap, 1, total)
            assert (t, status, h) == (total, ST_OVERFLOW, hits) and bool((out == -1).all())
            t, status, h, out = scan(passes, m, img, n, cap, 0, total)
            assert (t, status, h) == (total, ST_OVERFLOW, hits)
            assert torch.equal(out[:cap], want[:cap]) and bool((out[cap:] == -1).all())
        for part in (0, 1):
            t, status, h, out = scan(passes, m, img, n, total, part, total)
            assert (t, status, h) == (total, 0, hits) and torch.equal(out, want)


def fragments(passes, m, devs, sizes, mask_tiles, cap, room):
    """(total, status, first triple of each image, output as int64[room, 2], -1 where nothing was written)."""
    out = torch.full((room, 2), -1, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    n, u64, vp = len(devs), ctypes.c_uint64, ctypes.c_void_p
    h = (u64 * (2 + n))()
    rc = passes.passes_fragments(vp(m.handle), (vp * n)(*[d.data_ptr() for d in devs]), (u64 * n)(*sizes), ctypes.c_uint32(n),
                                 u64(mask_tiles), u64(cap), vp(out.data_ptr()), h)
    assert rc == 0
    return int(h[0]), int(h[1]) & 0xFFFFFFFF, [int(x) for x in h[2:]], out


def fragment_case(sig):
    """Three images (one without a match) of several tiles and a file of which fragments are planted, some
    with two master copies; the master file."""
    rng = np.random.default_rng(sig)
    file = rng.integers(0, 256, 64 * 50, dtype=np.uint8)
    file = np.concatenate([file, file[:640]])
    images = []
    for size, plants in ((30_011, 40), (9_000, 0), (70_000, 60)):
        img = rng.integers(0, 256, size, dtype=np.uint8)
        for w in rng.integers(0, (size - 64) // 4, plants):
            k = int(rng.integers(0, 60))
            img[4 * w:4 * w + 64] = file[64 * k:64 * k + 64]
        images.append(img)
    return images, file


@pytest.mark.parametrize("sig", [0, 1, 2])
def test_fragments_without_room(cv, passes, sig):
    """Without room for every triple of all images none is written, and it is said so."""
    images, file = fragment_case(sig)
    devs = [torch.from_numpy(x).cuda() for x in images]
    with cv.master_build([file], signature=sig, unit=cv.CV_UNIT_FRAGMENT) as m:
        with cv.scan(m, devs, keep_on_device=True) as r:
            want = torch.cat([torch.as_tensor(r.matches(i), device="cuda").view(torch.int64).clone() for i in (0, 2)])
        total = want.shape[0]
        assert total > 40
        for cap in (0, 1, total - 1, total, total + 5):
            t, status, first, out = fragments(passes, m, devs, [x.size for x in images], 1 << 22, cap, total)
            assert t == total and status == (0 if cap >= total else ST_OVERFLOW)
            assert torch.equal(out, want) if cap >= total else bool((out == -1).all())


@pytest.mark.parametrize("sig", [0, 1, 2])
@pytest.mark.parametrize("mask_tiles", [0, 1, 2, 9, 12, 1 << 20])
def test_hit_lists_beyond_their_masks(cv, passes, sig, mask_tiles):
    """Masks for none, some (ending within an image, at its first tile, before it) or all of the listed tiles:
    the windows of the others are looked up again. The images' first triples are right as well."""
    images, file = fragment_case(sig)
    devs = [torch.from_numpy(x).cuda() for x in images]
    want = [oracle.frag_match(x, [file]) for x in images]
    total = sum(w.size for w in want)
    for kw in ({}, {"bloom_bits_per_key": 0}, {"layout": cv.CV_LAYOUT_SORTED}):
        with cv.master_build([file], signature=sig, unit=cv.CV_UNIT_FRAGMENT, **kw) as m:
            t, status, first, out = fragments(passes, m, devs, [x.size for x in images], mask_tiles, total, total)
        assert (t, status) == (total, 0)
        assert first[:3] == [0, want[0].size, want[0].size]
        got = out.cpu().numpy()
        every = np.concatenate(want)
        assert np.array_equal(got[:, 0], every["disk_sector"].astype(np.int64))
        assert np.array_equal(got[:, 1] >> 32, every["file_sector"].astype(np.int64))
