"""The work that is timed: scans of disk images against tables of known files, and table builds.

Every case is one call (or one short sequence of calls) that a program using the library makes,
through the Python binding of the C ABI. Inputs are synthetic and made on the GPU: image sectors
are 70% uniform random bytes, 15% zero, 15% text of a 2,000-word vocabulary; master files are
random bytes of log-uniform size (8 KiB to 1 MiB); a share of the image's 4 KiB clusters carries
clusters of the master files, and the first 1 to 4 sectors of a tenth of those are overwritten.
Fragment workloads plant small files of 1 to 16 KiB at 4-byte offsets.
"""
import math

import numpy as np
import torch

from paper_0901_1307_gb300 import cv

SECTOR = 512
CLUSTER = 8                # sectors of a 4 KiB cluster
FRAG = 64
MD5, MD5_NOPAD, DJB2, CRC64 = cv.CV_SIG_MD5, cv.CV_SIG_MD5_NOPAD, cv.CV_SIG_DJB2_64, cv.CV_SIG_CRC64
_CHUNK = 1 << 20           # sectors generated at a time
_OPS = {MD5: 2852, MD5_NOPAD: 2560, DJB2: 128 * 5, CRC64: 128 * 10}  # integer operations per sector
_FRAG_OPS = {MD5: 690, MD5_NOPAD: 385, DJB2: 31}                     # per window


def _scan(name, image_bytes, master_sectors, **kw):
    c = dict(name=name, kind="scan", image_bytes=image_bytes, master_sectors=master_sectors, signature=MD5,
             host=False, keep=False, density=0.01, max_load=0.5, bloom=16, layout=cv.CV_LAYOUT_HASH, cluster=False)
    c.update(kw)
    return c


def listed():
    return [
        # a network-stream chunk that has just landed in a device buffer: latency and launches
        _scan("chunk_64k", 64 << 10, 1 << 20, density=0.05),
        # a small image handed over in pinned host memory, against a small case's files: the copy,
        # the scan and the matches back on the host
        _scan("host_64m", (64 << 20) + 100, 40803, host=True, density=0.12),
        # one partition of a drive on the device, its length not a whole number of sectors; the
        # matches come back to the host
        _scan("image_1g", (1 << 30) + 7 * SECTOR + 13, 1 << 20),
        # a whole drive image, results left on the device: the benchmark's own workload
        _scan("image_32g", 32 << 30, 4194304, keep=True, density=0.0156),
        # the same sectors without the padding block (Section 2.1)
        _scan("nopad_4g", (4 << 30) - 3 * SECTOR, 1 << 20, signature=MD5_NOPAD, keep=True),
        # the paper's own signatures, every candidate confirmed byte for byte
        _scan("djb2_8g", 8 << 30, 4194304, signature=DJB2, keep=True),
        _scan("crc64_cluster_2g", (2 << 30) + 5 * SECTOR, 1 << 20, signature=CRC64, keep=True, cluster=True),
        # a table packed to 90% without a filter, its layout left to the library (Section 4.2)
        _scan("packed_table_4g", 4 << 30, 7549747, max_load=0.9, bloom=0, layout=cv.CV_LAYOUT_AUTO, keep=True),
        # many drives of uneven size against one table, one graph replay per pass
        dict(name="batch_16g", kind="batch", n_images=256, image_bytes=16 << 30, master_sectors=8388608,
             signature=MD5, density=0.01),
        # logos and small images embedded at any 4-byte offset (Section 5)
        dict(name="frag_djb2_1g", kind="fragments", image_bytes=(1 << 30) + 36, logos=2000, signature=DJB2),
        dict(name="frag_md5_256m", kind="fragments", image_bytes=256 << 20, logos=500, signature=MD5),
        # a new set of known files: the table is built, then a first small image goes through it
        dict(name="build_4m", kind="build", image_bytes=16 << 20, master_sectors=4194304, signature=MD5,
             density=0.05),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["scan"] * 6 + ["batch"] * 2 + ["fragments"] * 2 + ["build"] * 2)
    sig = rng.choice([MD5, MD5, MD5, MD5_NOPAD, DJB2, CRC64])
    if kind == "scan":
        host = rng.random() < 0.2
        bytes_ = _log(rng, 64 << 10, (256 << 20) if host else (16 << 30))
        masters = _log(rng, 1000, 8 << 20)
        packed = rng.random() < 0.3
        return dict(kind=kind, image_bytes=bytes_, master_sectors=masters, signature=sig, host=host,
                    keep=not host and rng.random() < 0.5, density=rng.choice([0.0001, 0.01, 0.1]),
                    max_load=0.9 if packed else 0.5, bloom=rng.choice([0, 16]) if packed else 16,
                    layout=rng.choice([cv.CV_LAYOUT_SORTED, cv.CV_LAYOUT_AUTO]) if packed else cv.CV_LAYOUT_HASH,
                    cluster=rng.random() < 0.25)
    if kind == "batch":
        n = _log(rng, 2, 512)
        return dict(kind=kind, n_images=n, image_bytes=_log(rng, max(16 << 20, n * (64 << 10)), 16 << 30),
                    master_sectors=_log(rng, 10000, 8 << 20), signature=sig, density=rng.choice([0.01, 0.1]))
    if kind == "fragments":
        fsig = rng.choice([MD5, MD5_NOPAD, DJB2, DJB2])
        logos = _log(rng, 20, 2000)
        return dict(kind=kind, image_bytes=max(_log(rng, 4 << 20, (2 << 30) if fsig == DJB2 else (256 << 20)),
                                               logos * (64 << 10)),
                    logos=logos, signature=fsig)
    return dict(kind=kind, image_bytes=_log(rng, 1 << 20, 64 << 20), master_sectors=_log(rng, 20000, 8 << 20),
                signature=sig, density=0.05)


# ------------------------------------------------------------------------------------ inputs
# How many files and planted clusters there are, and how large, is the case's (the number of
# matches is an output's length); all contents and positions are the seed's.
def _shape_rng(case):
    return np.random.default_rng([case["image_bytes"], case.get("master_sectors", 0), case.get("logos", 0)])


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _text(rng):
    """4 MiB of words, as 64-bit words on the GPU."""
    words = ["".join(map(chr, rng.integers(97, 123, size=rng.integers(2, 11)))) for _ in range(2000)]
    s = " ".join(words[k] for k in rng.integers(0, 2000, size=700000)).encode()[: 4 << 20]
    return torch.frombuffer(bytearray(s), dtype=torch.uint8).view(torch.int64).cuda()


def _background(n_sectors, seed, rng):
    """n_sectors sectors of the usual mix, as int64[n_sectors, 64]."""
    g = _gen(seed)
    text = _text(rng)
    img = torch.empty((n_sectors, 64), dtype=torch.int64, device="cuda")
    k = torch.arange(64, device="cuda")
    for a in range(0, n_sectors, _CHUNK):
        part = img[a:a + _CHUNK]
        part.random_(-2 ** 63, None, generator=g)
        u = torch.rand(part.shape[0], device="cuda", generator=g)
        part[u < 0.15] = 0
        t = torch.nonzero(u >= 0.85)[:, 0]
        off = torch.randint(0, text.numel() - 64, (t.numel(),), device="cuda", generator=g)
        part[t] = text[off[:, None] + k]
    return img


def _file_sectors(total, rng):
    """Whole sectors of master files of log-uniform 8 KiB to 1 MiB, `total` in all."""
    n = np.round(np.exp(rng.uniform(np.log(16), np.log(2048), size=total // 400 + 64))).astype(np.int64)
    while n.sum() < total:
        n = np.concatenate([n, n])
    last = int(np.searchsorted(np.cumsum(n), total))
    n = n[:last + 1]
    n[last] -= n.sum() - total
    return n


def _masters(case, seed, shape):
    total = case["master_sectors"]
    fsec = _file_sectors(total, shape)
    data = torch.empty((total, 64), dtype=torch.int64, device="cuda")
    data.random_(-2 ** 63, None, generator=_gen(seed + 1))
    base = np.concatenate([[0], np.cumsum(fsec)])
    files = np.stack([data.data_ptr() + base[:-1] * SECTOR, fsec * SECTOR], axis=1).astype(np.uint64)
    return data, files, fsec, base


def _plant_plan(n_sectors, density, fsec, base, shape, rng):
    """(image sector, file, file sector, master sector) of every planted sector that is left."""
    n_cl = n_sectors // CLUSTER
    count = max(1, round(density * n_cl))
    q = np.unique(rng.integers(0, n_cl, size=count + count // 4 + 64)) if count < n_cl // 4 else np.arange(n_cl)
    q = np.sort(rng.permutation(q)[:count])
    cl = np.cumsum((fsec + CLUSTER - 1) // CLUSTER)
    g = shape.integers(0, cl[-1], size=count)
    f = np.searchsorted(cl, g, side="right")
    c = g - np.concatenate([[0], cl])[f]
    over = np.where(shape.random(count) < 0.1, shape.integers(1, 5, size=count), 0)
    mix = rng.permutation(count)
    f, c, over = f[mix], c[mix], over[mix]
    k = np.arange(CLUSTER)
    i, s = q[:, None] * CLUSTER + k, c[:, None] * CLUSTER + k
    keep = (k >= over[:, None]) & (s < fsec[f][:, None])
    f = np.broadcast_to(f[:, None], s.shape)[keep]
    return i[keep], f, s[keep], base[f] + s[keep]


def _image(case, n_bytes, seed, data, fsec, base, shape, rng):
    """A device image of n_bytes with planted clusters (a uint8 tensor), and the plant plan."""
    n = n_bytes // SECTOR
    img = _background((n_bytes + SECTOR - 1) // SECTOR, seed + 2, rng)
    plan = _plant_plan(n, case["density"], fsec, base, shape, rng)
    at, src = torch.from_numpy(plan[0]).cuda(), torch.from_numpy(plan[3]).cuda()
    for a in range(0, at.numel(), _CHUNK):
        img[at[a:a + _CHUNK]] = data[src[a:a + _CHUNK]]
    return img.view(torch.uint8).reshape(-1)[:n_bytes], plan


def _build(case, files):
    return cv.master_build(files, max_load=case.get("max_load", 0.5), bloom_bits_per_key=case.get("bloom", 16),
                           signature=case["signature"], layout=case.get("layout", cv.CV_LAYOUT_HASH),
                           position_mode=cv.CV_POSITION_CLUSTER if case.get("cluster") else cv.CV_POSITION_ANY)


def _batch_sectors(case, shape):
    """Sectors of every image of a batch: log-uniform over a factor of 2,048, image_bytes in all."""
    w = np.exp(shape.uniform(0, np.log(2048), size=case["n_images"]))
    n = np.maximum(np.floor(w / w.sum() * (case["image_bytes"] // SECTOR)).astype(np.int64), 128)
    return n - n % CLUSTER


def _logos(case, shape, rng):
    """Small files as one byte array: (bytes, first byte of each, length of each)."""
    size = np.round(np.exp(shape.uniform(np.log(1024), np.log(16384), size=case["logos"]))).astype(np.int64)
    first = np.concatenate([[0], np.cumsum((size + 15) // 16 * 16)])
    data = rng.integers(0, 256, size=int(first[-1]), dtype=np.uint8)
    header = rng.integers(0, 256, size=128, dtype=np.uint8)
    for f in range(size.size):
        if shape.random() < 0.1:                      # a header that several files share
            data[first[f]:first[f] + 128] = header
        if size[f] >= 2048 and shape.random() < 0.2:  # a zero run: fragments the table leaves out
            z = int(first[f]) + FRAG * int(shape.integers(4, size[f] // FRAG - 4))
            data[z:z + FRAG * int(shape.integers(1, 4))] = 0
    return data, first, size


def _plant_logos(case, size, shape, rng):
    """(logo, byte offset) of every planted copy: half of the files, one to three times."""
    f = np.concatenate([np.nonzero(shape.random(size.size) < 0.5)[0], [0]])
    f = rng.permutation(np.repeat(f, shape.integers(1, 4, size=f.size)))
    region = case["image_bytes"] // f.size // 4 * 4
    return f, np.arange(f.size) * region + 4 * rng.integers(0, (region - size[f]) // 4 + 1)


# ------------------------------------------------------------------------------------- cases
def prepare(case, seed):
    rng, shape = np.random.default_rng(seed), _shape_rng(case)
    kind = case["kind"]
    state = dict(case=case)
    if kind == "fragments":
        data, first, size = _logos(case, shape, rng)
        dev = torch.from_numpy(data).cuda()
        files = np.stack([dev.data_ptr() + first[:-1], size], axis=1).astype(np.uint64)
        state["master"] = cv.master_build(files, signature=case["signature"], unit=cv.CV_UNIT_FRAGMENT)
        nb = case["image_bytes"]
        img = _background((nb + SECTOR - 1) // SECTOR, seed + 2, rng).view(torch.uint8).reshape(-1)[:nb]
        for f, o in zip(*_plant_logos(case, size, shape, rng)):
            img[o:o + size[f]] = dev[first[f]:first[f] + size[f]]
        state["image"] = img
        torch.cuda.synchronize()
        return state
    data, files, fsec, base = _masters(case, seed, shape)
    if kind == "batch":
        sectors = _batch_sectors(case, shape)
        whole, _ = _image(case, int(sectors.sum()) * SECTOR, seed, data, fsec, base, shape, rng)
        state["images"] = list(torch.split(whole, (sectors * SECTOR).tolist()))
        torch.cuda.synchronize()
        state["master"] = _build(case, files)
        state["batch"] = cv.batch_create(state["master"], state["images"])
        return state
    img, _ = _image(case, case["image_bytes"], seed, data, fsec, base, shape, rng)
    torch.cuda.synchronize()
    if kind == "build":
        state.update(image=img, data=data, files=files)
        return state
    state["master"] = _build(case, files)
    if case["host"]:
        pinned = torch.empty(img.numel(), dtype=torch.uint8, pin_memory=True)
        pinned.copy_(img)
        img = pinned
    state["image"] = img
    return state


def _host_rows(result):
    """Image 0's matches as int32[n, 4]: disk sector (two words), file, file sector."""
    return result.matches(0).view(np.int32).reshape(-1, 4)


def _device_rows(m):
    """Device matches as int64[n, 2]: disk sector, file + file sector * 2^32."""
    if m.n == 0:
        return torch.empty((0, 2), dtype=torch.int64, device="cuda")
    return torch.as_tensor(m, device="cuda").view(torch.int64)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "scan":
        r = cv.scan(state["master"], [state["image"]], keep_on_device=case["keep"])
        return _device_rows(r.matches(0)) if case["keep"] else _host_rows(r)
    if kind == "batch":
        b = state["batch"]
        b.run()
        n = b.wait()
        # the images' matches lie one after another in the batch's buffer
        first = next((m.ptr for m in map(b.matches, range(b.n_images)) if m.n), 0)
        return _device_rows(cv.DeviceMatches(first, n, b))
    if kind == "fragments":
        return _host_rows(cv.scan(state["master"], [state["image"]]))
    with _build(case, state["files"]) as m, cv.scan(m, [state["image"]]) as r:
        info = m.info()
        return [_host_rows(r)] + [info[k] for k in ("n_sectors", "n_kept", "n_unique", "n_slots", "bloom_bytes")]


def _expected(case, seed):
    """Rows (disk sector, file, file sector) that the inputs of prepare(case, seed) hold."""
    rng, shape = np.random.default_rng(seed), _shape_rng(case)
    if case["kind"] == "fragments":
        data, first, size = _logos(case, shape, rng)
        nfr = size // FRAG
        f = np.repeat(np.arange(size.size), nfr)
        j = np.arange(f.size) - np.repeat(np.cumsum(nfr) - nfr, nfr)
        rows = np.stack([data[first[a] + FRAG * b:first[a] + FRAG * b + FRAG] for a, b in zip(f, j)])
        fill = (rows == rows[:, :1]).all(axis=1)
        _, key = np.unique(rows.view("V%d" % FRAG)[:, 0], return_inverse=True)
        members = {}
        for x in np.nonzero(~fill)[0]:
            members.setdefault(int(key[x]), []).append((int(f[x]), int(j[x])))
        _text_only(rng)
        at = np.cumsum(nfr) - nfr
        out = [(o // 4 + 16 * b, *m) for g, o in zip(*_plant_logos(case, size, shape, rng)) for b in range(nfr[g])
               if not fill[at[g] + b] for m in members[int(key[at[g] + b])]]
        return np.array(sorted(out), dtype=np.int64).reshape(-1, 3)
    fsec = _file_sectors(case["master_sectors"], shape)
    base = np.concatenate([[0], np.cumsum(fsec)])
    sectors = _batch_sectors(case, shape) if case["kind"] == "batch" else np.array([case["image_bytes"] // SECTOR])
    _text_only(rng)
    i, f, s, _ = _plant_plan(int(sectors.sum()), case["density"], fsec, base, shape, rng)
    start = np.concatenate([[0], np.cumsum(sectors)])
    i = i - start[np.searchsorted(start, i, side="right") - 1]  # within its image
    if case.get("cluster"):
        ok = i % CLUSTER == s % CLUSTER
        i, f, s = i[ok], f[ok], s[ok]
    return np.stack([i, f, s], axis=1).astype(np.int64)


def _text_only(rng):
    """Draws what _text draws."""
    for _ in range(2000):
        rng.integers(97, 123, size=rng.integers(2, 11))
    rng.integers(0, 2000, size=700000)


def exact(case, seed):
    """The matches that the inputs hold by construction: master sectors are random and distinct."""
    e = _expected(case, seed)
    if case["kind"] == "batch" or case.get("keep"):
        return torch.from_numpy(np.stack([e[:, 0], e[:, 1] | (e[:, 2] << 32)], axis=1))
    rows = np.stack([e[:, 0] & 0xFFFFFFFF, e[:, 0] >> 32, e[:, 1], e[:, 2]], axis=1).astype(np.uint32).view(np.int32)
    if case["kind"] != "build":
        return rows
    m = case["master_sectors"]
    slots = max(2, 1 << (int(m / 0.5)).bit_length())
    return [rows, m, m, m, slots, 32 << max(0, ((m * 16 + 255) // 256 - 1).bit_length())]


def work(case):
    """Bytes: the image (or the master files) read once, matches and tables written once.
    Operations: the integer operations of the signatures."""
    nb, sig = case["image_bytes"], case["signature"]
    if case["kind"] == "fragments":
        return {"bytes": nb + 16 * 60 * case["logos"], "flops": (nb // 4) * _FRAG_OPS[sig]}
    out = int(16 * case["density"] * (nb // SECTOR))
    if case["kind"] != "build":
        return {"bytes": nb + out, "flops": (nb // SECTOR) * _OPS[sig]}
    m = case["master_sectors"]
    # files read; a 32-byte record per key, an 8-byte posting and 16 filter bits written
    return {"bytes": nb + out + m * (SECTOR + 32 + 8 + 2), "flops": (nb // SECTOR + m) * _OPS[sig]}
