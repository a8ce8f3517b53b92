"""A surface update that gets no memory for one of its arrays leaves nothing
half-built: the surface holds the last update's mesh, or none until the next
update, which then rebuilds it."""
import ctypes as C

import numpy as np
import pytest

import bm_inputs as bi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import torch
    assert torch.cuda.is_available()
    import paper_2609_27342_gb300 as p
    from paper_2609_27342_gb300 import build
    build.build()
    p.load()
    return p


class _Limited:
    """bm_alloc over PyTorch's caching allocator that refuses the request after `left` more."""

    def __init__(self):
        import torch
        from paper_2609_27342_gb300 import _abi as A
        self.left = -1      # no limit

        def alloc(nbytes, stream, ctx):
            if self.left == 0:
                self.left = -1
                return None
            self.left -= self.left > 0
            return int(torch.cuda.caching_allocator_alloc(int(nbytes), torch.cuda.current_device(), stream or 0))

        def free(ptr, stream, ctx):
            if ptr:
                torch.cuda.caching_allocator_delete(int(ptr))

        self._fns = A.ALLOC_FN(alloc), A.FREE_FN(free)
        self.struct = A.Alloc(*self._fns, None)


@pytest.mark.parametrize("granted", [0, 1])   # the vertices', then the triangles' request is refused
def test_refused_array_leaves_no_half_built_surface(pkg, granted):
    from paper_2609_27342_gb300 import _abi as A
    from paper_2609_27342_gb300.surface import Surface
    sc = bi.Scene(X=bi.lattice_cuboid((0.05, 0.03, 0.03), 5e-3), dx=5e-3)
    al = _Limited()
    s = pkg.Scene(sc, allocator=al)
    f = Surface(s)
    small = f.update()
    old = f.read()
    # cell-wide columns of eight codes: many times the vertices
    q = np.floor(sc.X / 5e-3).astype(int)
    bits = [(q[:, 0] >> 0) & 1, (q[:, 1] >> 0) & 1, (q[:, 2] >> 0) & 1]
    m1 = sum(b << k for k, b in enumerate(bits)).astype(np.uint32)
    m2 = (7 - m1).astype(np.uint32)
    s.write(mask1=m1, mask2=m2)
    al.left = granted
    with pytest.raises(A.BMError) as e:
        f.update()
    assert e.value.code == A.E_OOM and al.left == -1
    left = f.read()
    if granted == 0:   # the vertices stayed where they were
        assert (f.n_vertices, f.n_triangles) == small
        for k in ("reference", "triangles"):
            assert np.array_equal(left[k], old[k]), k
        f.update(rebuild=False)     # and can be moved on
        assert np.array_equal(f.read()["triangles"], old["triangles"])
    else:
        assert (f.n_vertices, f.n_triangles) == (0, 0) and len(left["vertices"]) == 0
    big = f.update(rebuild=granted == 0)
    got = f.read()
    g = Surface(s)
    assert g.update() == big and big[0] > 2 * small[0]
    want = g.read()
    for k in want:
        assert np.array_equal(got[k], want[k]), k
    f.close()
    g.close()
    s.close()
