"""Which form of the general brick kernels a set of scenes takes changes no bit.

Sparse sets: many one-brick scenes of few particles take the one-group forms at
a brick count where fuller ones take several groups; each scene must come out
as on its own, where it takes several.  Occupancy variants: a set with a larger
body runs the one-group forms at the variant's resident CTAs.
"""
import numpy as np
import pytest

import bm_inputs as bi

pytestmark = pytest.mark.gpu

DX = 5e-3
FIELDS = ("x", "v", "F", "D", "ut", "mask1", "mask2")


@pytest.fixture(scope="module")
def pkg():
    import torch
    assert torch.cuda.is_available()
    import paper_2609_27342_gb300 as p
    from paper_2609_27342_gb300 import build
    build.build()
    p.load()
    return p


def _scene(cells, per_axis=(2, 2, 2), jitter=0.2, blade=True, seed=0, **kw):
    X = bi.lattice_cuboid([c * DX for c in cells], DX, per_axis, jitter=jitter, seed=seed)
    size = X.max(0) - X.min(0) + DX
    # the edge stands in the top layer: contact, reaction and labels from the first substeps
    edge = (X[:, 0].mean() + 2e-4, X[:, 1].mean(), X[:, 2].max() - 0.2 * DX)
    b = bi.Blade(pose_x=tuple(float(t) for t in edge), half_length=float(size.max()),
                 segments=[bi.Segment(40, v=(0.0, 0.0, -1.5), omega=(0.5, 2.0, -1.0), cut_id=0)]) if blade else None
    return bi.Scene(X=X, dx=DX, origin=(-DX / 2,) * 3, V0=DX ** 3 / 8, dt=1e-4, E=1e5, nu=0.3, blade=b, **kw)


def _state(n, seed):
    rng = np.random.default_rng(seed)
    return dict(v=(0.3 * rng.standard_normal((n, 3))).astype(np.float32),
                F=(np.eye(3).ravel() + 0.02 * rng.standard_normal((n, 9))).astype(np.float32))


def _batch(pkg, specs):
    fp = [pkg.footprint(q) for q in specs]
    b = pkg.Batch(max_particles=sum(f[0] for f in fp), max_nodes=sum(f[1] for f in fp), max_scenes=len(specs),
                  max_bricks=sum(f[2] for f in fp))
    return b, sum(f[0] for f in fp), sum(f[2] for f in fp)


def test_sparse_set_equals_the_scenes_alone_bitwise(pkg):
    specs = [_scene((1, 1, 1), seed=i) if i % 3 else _scene((3, 2, 2), seed=i) for i in range(160)]
    b, n, bricks = _batch(pkg, specs)
    assert 152 < bricks <= 4 * 152 and n / bricks < 128
    ss = [pkg.Scene.in_batch(b, q) for q in specs]
    for i, s in enumerate(ss):
        s.write(**_state(s.n, i))
    b.step(8)
    for i in (0, 1, 78, 159):
        s = pkg.Scene(specs[i])
        s.write(**_state(s.n, i))
        s.step(8)
        want, got = s.read(*FIELDS), ss[i].read(*FIELDS)
        for k in FIELDS:
            assert np.array_equal(got[k], want[k]), (i, k)
        assert np.array_equal(ss[i].tool_wrench(), s.tool_wrench())
        assert ss[i].info().error_bits == 0
        s.close()
    for s in ss:
        s.close()
    b.close()


# 12 codes: more than the slot tables hold, and tiles beyond the slot window
@pytest.mark.parametrize("cells,per_axis,codes,kw", [
    ((9, 5, 6), (2, 2, 2), 1, {}), ((7, 5, 3), (4, 2, 2), 1, dict(jitter=0.0)),
    ((9, 5, 6), (2, 2, 2), 1, dict(yield_stress=2e3, viscosity=5.0)),
    ((7, 5, 3), (4, 2, 2), 1, dict(yield_stress=2e3, viscosity=5.0)),
    ((4, 4, 4), (2, 2, 2), 12, dict(blade=False)), ((4, 4, 4), (4, 2, 2), 12, dict(blade=False)),
])
def test_occupancy_variants_agree_bitwise(pkg, cells, per_axis, codes, kw):
    sc = _scene(cells, per_axis, **kw)
    filler = _scene((42, 42, 42), (1, 1, 1), blade=False)
    b, n, bricks = _batch(pkg, [sc, filler])
    assert bricks > 4 * 152
    s, f = pkg.Scene.in_batch(b, sc), pkg.Scene.in_batch(b, filler)
    q = np.floor(sc.X / DX).astype(int)
    code = (q[:, 0] % 4 + 4 * (q[:, 1] % 3)) * (codes > 1)    # columns of cells; 0: none, odd / even: side 1 / 2 of a cut
    bit = 1 << (1 + (code + 1) // 2)
    s.write(mask1=np.where(code % 2 == 1, bit, 0).astype(np.uint32),
            mask2=np.where((code % 2 == 0) & (code > 0), bit, 0).astype(np.uint32), **_state(s.n, 3))
    cut = f.spec.X[:, 0] < f.spec.X[:, 0].mean()     # several codes in some of its bricks
    f.write(mask1=np.where(cut, 2, 0).astype(np.uint32), mask2=np.where(cut, 0, 2).astype(np.uint32), **_state(f.n, 4))
    ck = s.checkpoint(), f.checkpoint()
    want = None
    # default, one other choice of each kernel, and the two others of all three
    for variant in (0, 1, 2, 3, 6, 9, 18, 13, 26):
        s.restore(ck[0])
        f.restore(ck[1])
        b.set_tiles(4, 128, variant)
        b.step(8)
        got = [g.read(*FIELDS) for g in (s, f)] + [s.tool_wrench() if codes == 1 else 0,
                                                   s.info().error_bits, f.info().error_bits]
        assert got[3] == 0 and got[4] == 0
        if want is None:
            want = got
            assert codes > 1 or (np.any(want[2] != 0) and np.any(want[0]["mask1"] | want[0]["mask2"]))
        for i in (0, 1):
            for k in FIELDS:
                assert np.array_equal(got[i][k], want[i][k]), (variant, i, k)
        assert np.array_equal(got[2], want[2]), variant
    s.close()
    f.close()
    b.close()
