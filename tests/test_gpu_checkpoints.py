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


@pytest.mark.parametrize("where", ["device", "device+4", "device+1", "pinned", "managed"])
def test_any_buffer_holds_a_checkpoint(pkg, where):
    """Device memory in one launch, by 16-byte words, 4-byte words or bytes as
    its alignment allows; other memory section by section."""
    import torch
    from paper_2609_27342_gb300 import _abi as A
    sc = bi.single_cut_cuboid(size=(0.04, 0.02, 0.02), edge_z0=0.0201, speed=1.0, n_down=100)
    s = pkg.Scene(sc)
    s.step(20)
    n = s.checkpoint_size()
    keep = None
    if where == "managed":
        rt = C.CDLL("libcudart.so.13")
        p = C.c_void_p()
        assert rt.cudaMallocManaged(C.byref(p), C.c_size_t(n), C.c_uint(1)) == 0
        ptr, on_device = p.value, 1
    else:
        off = int(where.partition("+")[2] or 0)
        keep = torch.empty(n + 256, dtype=torch.uint8, device="cpu", pin_memory=True) if where == "pinned" else \
            torch.empty(n + 256, dtype=torch.uint8, device="cuda")
        keep.fill_(0x5a)
        torch.cuda.synchronize()
        ptr, on_device = keep.data_ptr() + off, int(keep.is_cuda)
    L = A.load()
    A.check(L.bm_checkpoint_save(s.handle, C.c_void_p(ptr), on_device))
    if keep is not None:    # nothing is written outside the checkpoint
        assert bool((keep[:off] == 0x5a).all()) and bool((keep[off + n:] == 0x5a).all())
    s.step(6)
    want = s.read("x", "v", "F", "D", "ut", "mask1", "mask2")
    tool = s.tool_state()
    s.step(3)
    A.check(L.bm_checkpoint_restore(s.handle, C.c_void_p(ptr), on_device))
    s.step(6)
    for k, v in s.read(*want).items():
        assert np.array_equal(v, want[k]), k
    assert np.array_equal(s.tool_state(), tool)
    s.close()
    if where == "managed":
        assert rt.cudaFree(p) == 0


def test_surface_read_into_device_memory(pkg):
    import torch
    from paper_2609_27342_gb300.surface import Surface
    s = pkg.Scene(bi.Scene(X=bi.lattice_cuboid((0.03, 0.02, 0.02), 5e-3), dx=5e-3))
    f = Surface(s)
    nv, nt = f.update()
    want = f.read()
    v = torch.zeros(nv + 1, 3, device="cuda")
    t = torch.zeros(nt, 3, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    f.read_into(v[1:], t)
    assert np.array_equal(v[1:].cpu().numpy(), want["vertices"]) and bool((v[0] == 0).all())
    assert np.array_equal(t.cpu().numpy(), want["triangles"])
    f.close()
    s.close()
