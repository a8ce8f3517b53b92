"""Checkpoints: what a restore reads before it knows the buffer to be the
scene's, and what it leaves to the scene (its place and its stop substep)."""
import ctypes as C
import mmap

import numpy as np
import pytest

import bm_inputs as bi

pytestmark = pytest.mark.gpu

HEADER = 48     # bytes of the checkpoint header (magic, four int64, two int32)


@pytest.fixture(scope="module")
def pkg():
    import torch
    assert torch.cuda.is_available()
    import paper_2609_27342_gb300 as p
    from paper_2609_27342_gb300 import build
    build.build()
    p.load()
    return p


def test_short_buffer_without_a_checkpoint_is_refused(pkg):
    """The C entry is told no size, so it may read no further than the header
    of a buffer that holds no checkpoint of the scene."""
    from paper_2609_27342_gb300 import _abi as A
    sc = bi.Scene(X=bi.lattice_cuboid((0.02, 0.01, 0.01), 5e-3), dx=5e-3)
    s = pkg.Scene(sc)
    before = s.read("x", "v", "F")
    good = s.checkpoint(device=False)
    # the last readable bytes ahead of a page without access
    page = mmap.PAGESIZE
    area = mmap.mmap(-1, 2 * page)
    addr = C.addressof(C.c_char.from_buffer(area))
    libc = C.CDLL(None, use_errno=True)
    assert libc.mprotect(C.c_void_p(addr + page), C.c_size_t(page), 0) == 0
    short = addr + page - HEADER
    L = A.load()
    for head in (bytes(HEADER), good[:8].tobytes() + bytes(HEADER - 8)):   # no magic; the magic and no scene of this size
        C.memmove(short, head, HEADER)
        assert L.bm_checkpoint_restore(s.handle, C.c_void_p(short), 0) == A.E_INVALID
    after = s.read("x", "v", "F")
    for k in before:
        assert np.array_equal(before[k], after[k]), k
    s.step(2)
    s.restore(good)
    assert np.array_equal(s.read("x")["x"], before["x"])
    s.close()
    assert libc.mprotect(C.c_void_p(addr + page), C.c_size_t(page), mmap.PROT_READ | mmap.PROT_WRITE) == 0


@pytest.mark.parametrize("device", [True, False])
def test_restore_keeps_place_and_stop_substep(pkg, device):
    """Saved alone, restored as the second scene of a batch: the state is the
    saved one and the ranges are the batch's; a stop substep set since then
    still holds, on both sides of the restored substep."""
    sc = bi.single_cut_cuboid(size=(0.04, 0.02, 0.02), edge_z0=0.0201, speed=1.0, n_down=100)
    s, other = pkg.Scene(sc), pkg.Scene(sc)
    s.step(20)
    ck = s.checkpoint(device=device)
    s.step(6)
    want = s.read("x", "v", "F", "mask1", "mask2")
    tool = s.tool_state()
    s.step(5)
    fp = pkg.footprint(sc)
    b = pkg.Batch(max_particles=2 * fp[0], max_nodes=2 * fp[1], max_scenes=2, max_bricks=2 * fp[2])
    b.add(other)
    b.add(s)
    s.set_stop(26)
    s.restore(ck)                 # six substeps to go
    b.step(10)
    assert s.info().step == 26 and other.info().step == 10
    for k, v in s.read("x", "v", "F", "mask1", "mask2").items():
        assert np.array_equal(v, want[k]), k
    assert np.array_equal(s.tool_state(), tool)
    s.set_stop(15)
    s.restore(ck)                 # beyond the stop: stays as restored
    b.step(3)
    assert s.info().step == 20 and other.info().step == 13
    s.set_stop(-1)
    s.restore(ck)
    b.step(6)
    for k, v in s.read("x", "v", "F", "mask1", "mask2").items():
        assert np.array_equal(v, want[k]), k
    s.close()
    other.close()
    b.close()
