"""A batch that puts its own filter in front of a table without one looks the sectors up behind it as a
table built with a filter does, in the slots: it does not read the tags, which are for lookups of every
sector. Shown with a table whose tags are cleared."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_0901_1307_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cv(cuda_device):
    import __graft_entry__

    __graft_entry__.build()
    from paper_0901_1307_gb300 import cv as cvmod

    return cvmod


def table_arrays(cv, master):
    """(slots, tags) of a table's device view."""
    view, dev = (ctypes.c_uint64 * 64)(), ctypes.c_int()
    fn = getattr(cv.load(), "_ZN3cvk11master_viewEPK9cv_masterPNS_9TableViewEPi")
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p]
    assert fn(master.handle, view, ctypes.byref(dev)) == cv.CV_OK
    return view[0], view[6]


@pytest.mark.parametrize("sig", [0, 3])
@pytest.mark.parametrize("sorted_copy", [False, True])
def test_own_filter_looks_in_the_slots(cv, sig, sorted_copy):
    plan = synth.config_plan("small:16000:30:91")
    img, files = plan.image_host(), plan.masters_host()
    want = oracle.match_hash(img, files)
    dev = torch.from_numpy(img).cuda()
    with cv.master_build(files, signature=sig, bloom_bits_per_key=0) as m:
        slots, tags = table_arrays(cv, m)
        n = m.info()["n_slots"]
        assert n >= 64 and tags == slots + 32 * n
        clear = type("T", (), {"__cuda_array_interface__": {"shape": (n,), "typestr": "|u1", "data": (tags, False),
                                                           "version": 3, "strides": None}})()
        torch.as_tensor(clear, device="cuda").zero_()
        torch.cuda.synchronize()
        with cv.scan(m, [dev]) as r:
            assert r.count(0) == 0  # a scan of the table itself walks the tags
        with cv.batch_create(m, [dev], bloom=cv.CV_BATCH_BLOOM_ON, sorted_copy=sorted_copy) as b:
            b.run()
            assert b.wait() == want.size
            assert np.array_equal(cv.device_matches_to_numpy(b.matches(0)), want)
