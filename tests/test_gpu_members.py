"""A scene of a batch after another member was destroyed: what rebuilds its slot
tables must walk the scene's own bricks, not the list from before.

The scene is restored or relabelled right after the destruction, stepped, and
compared bit for bit with the same scene on its own.
"""
import numpy as np
import pytest

import bm_inputs as bi

pytestmark = pytest.mark.gpu

DX = 5e-3
FIELDS = ("x", "v", "F", "mask1", "mask2")


@pytest.fixture(scope="module")
def pkg():
    import torch
    assert torch.cuda.is_available()
    import paper_2609_27342_gb300 as p
    from paper_2609_27342_gb300 import build
    build.build()
    p.load()
    return p


def _scene(cells, jitter):
    X = bi.lattice_cuboid([c * DX for c in cells], DX, jitter=jitter)
    return bi.Scene(X=X, dx=DX, origin=(-DX / 2,) * 3, V0=DX ** 3 / 8, dt=1e-4, E=1e5, nu=0.3)


@pytest.mark.parametrize("jitter", [0.0, 0.1])
@pytest.mark.parametrize("how", ["restore", "relabel"])
def test_rebuild_after_a_member_was_destroyed(pkg, how, jitter):
    rng = np.random.default_rng(2)
    gone, sc = _scene((13, 9, 9), jitter), _scene((9, 6, 5), jitter)   # the first has more bricks
    n = len(sc.X)
    side = sc.X[:, 0] < sc.X[:, 0].mean()
    state = dict(v=(0.3 * rng.standard_normal((n, 3))).astype(np.float32),
                 F=(np.eye(3).ravel() + 0.02 * rng.standard_normal((n, 9))).astype(np.float32))
    cut = dict(mask1=np.where(side, 1, 0).astype(np.uint32), mask2=np.where(side, 0, 1).astype(np.uint32))
    got = []
    for batched in (True, False):
        s = pkg.Scene(sc)
        if batched:
            fp = [pkg.footprint(q) for q in (gone, sc)]
            b = pkg.Batch(max_particles=sum(f[0] for f in fp), max_nodes=sum(f[1] for f in fp), max_scenes=2,
                          max_bricks=sum(f[2] for f in fp))
            a = pkg.Scene(gone)
            b.add(a)
            b.add(s)
        s.write(**state)
        if how == "restore":      # back to the labelled state from one without labels
            s.write(**cut)
            ck = s.checkpoint()
            s.write(**{k: np.zeros_like(m) for k, m in cut.items()})
        if batched:
            a.close()
        if how == "restore":
            s.restore(ck)
        else:
            s.write(**cut)
        s.step(4)
        if batched:
            b.step(4)
        else:
            s.step(4)
        got.append((s.read(*FIELDS), s.info().n_slots, s.info().error_bits))
        s.close()
        if batched:
            b.close()
    for k in FIELDS:
        assert np.array_equal(got[0][0][k], got[1][0][k]), k
    assert got[0][1:] == got[1][1:]
