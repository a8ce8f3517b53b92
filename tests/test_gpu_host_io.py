"""State read into and written from host memory: fields go through one staging
buffer of the scene's world, or an allocation where they are too long for it,
and threads that read and write different scenes of a batch take turns."""
import threading

import numpy as np
import pytest

import bm_inputs as bi

pytestmark = pytest.mark.gpu

DX = 5e-3


@pytest.fixture(scope="module")
def pkg():
    import torch
    assert torch.cuda.is_available()
    import paper_2609_27342_gb300 as p
    from paper_2609_27342_gb300 import build
    build.build()
    p.load()
    return p


def _scene(cells, **kw):
    return bi.Scene(X=bi.lattice_cuboid([c * DX for c in cells], DX), dx=DX, **kw)


# one cell; F at the 4 MiB staging buffer's end and beyond it (36 B a particle);
# the pair history (192 B a particle) within it and beyond
@pytest.mark.parametrize("cells,kw", [((1, 1, 1), {}), ((48, 16, 18), {}), ((48, 16, 19), {}), ((48, 16, 20), {}),
                                      ((4, 4, 4), dict(pair_contact=True)), ((14, 14, 16), dict(pair_contact=True))])
def test_host_and_device_io_agree(pkg, cells, kw):
    import torch
    sc = _scene(cells, **kw)
    n = sc.n
    rng = np.random.default_rng(1)
    state = dict(x=(sc.X + 1e-4 * rng.standard_normal((n, 3))).astype(np.float32),
                 v=rng.standard_normal((n, 3)).astype(np.float32),
                 F=(np.eye(3).ravel() + 0.01 * rng.standard_normal((n, 9))).astype(np.float32),
                 D=rng.random(n).astype(np.float32), ut=rng.standard_normal((n, 3)).astype(np.float32),
                 mask1=rng.integers(0, 2, n).astype(np.uint32) << 1, mask2=np.zeros(n, np.uint32))
    s = pkg.Scene(sc)
    s.write(**state)
    got = s.read(*state)
    for k in state:
        assert np.array_equal(got[k], state[k]), k
    dev = {k: torch.empty(v.shape, dtype=torch.from_numpy(v.view(np.int32 if v.dtype == np.uint32 else v.dtype)).dtype,
                          device="cuda") for k, v in state.items()}
    s.read_device(dev)
    for k in state:
        assert np.array_equal(dev[k].cpu().numpy().view(state[k].dtype), state[k]), k
    code = s.read("code")["code"]
    assert np.array_equal(code, np.where(state["mask1"] > 0, 3, 0))
    if kw:
        s.step(1)
        h = s.read("pair_partner", "pair_u")
        assert h["pair_partner"].shape == (n, 16) and h["pair_partner"].max() < n
    s.close()


def test_threads_read_and_write_scenes_of_one_batch(pkg):
    sc = _scene((10, 8, 8))
    fp = pkg.footprint(sc)
    k = 4
    b = pkg.Batch(max_particles=k * fp[0], max_nodes=k * fp[1], max_scenes=k, max_bricks=k * fp[2])
    ss = [pkg.Scene.in_batch(b, sc) for _ in range(k)]
    bad = []

    def work(i):
        import torch
        torch.cuda.set_device(0)
        rng = np.random.default_rng(i)
        for _ in range(30):
            v = rng.standard_normal((sc.n, 3)).astype(np.float32)
            ss[i].write(v=v)
            if not np.array_equal(ss[i].read("x", "v")["v"], v):
                bad.append(i)

    th = [threading.Thread(target=work, args=(i,)) for i in range(k)]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not bad
    for s in ss:
        s.close()
    b.close()
