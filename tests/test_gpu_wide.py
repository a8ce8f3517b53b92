"""Brick kernels of sets of few bricks against those of larger sets, bit for bit.

A scene stepped alone takes the forms with several groups of threads per
brick; in a batch filled up with a larger body it takes the one-group forms
and the slot rebuild's other launches.  Every sum has the same terms in the
same order in both, so the scene must come out with the same bits.
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


def _lattice(cells, k):
    ax = [((np.arange(n * m) + 0.5) / m) * DX for n, m in zip(cells, k)]
    return np.stack(np.meshgrid(*ax, indexing="ij"), -1).reshape(-1, 3)


def _scene(X, blade, mass=0.0, **kw):
    size = X.max(0) - X.min(0) + DX
    # the edge stands in the top layer: contact, reaction and labels from the first substeps
    edge = (X[:, 0].mean() + 2e-4, X[:, 1].mean(), X[:, 2].max() - 0.2 * DX)
    b = bi.Blade(pose_x=tuple(float(t) for t in edge), half_length=float(size.max()),
                 mass=mass, inertia=tuple(4e-5 * mass * np.diag((1.0, 2.0, 3.0)).ravel()), rigid_interval=2 if mass else 1,
                 segments=[bi.Segment(40, v=(0.0, 0.0, -1.5), omega=(0.5, 2.0, -1.0), cut_id=0)]) if blade else None
    return bi.Scene(X=X, dx=DX, origin=(-DX / 2,) * 3, V0=DX ** 3 / 8, dt=1e-4, E=1e5, nu=0.3, blade=b, **kw)


# one cell, part of a brick, a ragged body of several bricks; 1, 8 and 16
# particles per cell, on a lattice and off it; 1, 3 and 12 codes
@pytest.mark.parametrize("cells,k,jitter,codes,kw", [
    ((1, 1, 1), (1, 1, 1), 0.0, 1, {}), ((9, 5, 6), (2, 2, 2), 0.0, 3, {}), ((4, 4, 4), (2, 2, 2), 0.0, 12, {}),
    ((9, 5, 6), (2, 2, 2), 0.1, 3, {}), ((4, 4, 4), (2, 2, 2), 0.1, 12, {}), ((7, 5, 3), (4, 2, 2), 0.0, 3, {}),
    ((7, 5, 3), (2, 2, 2), 0.1, 2, dict(yield_stress=2e3, viscosity=5.0)),
    ((9, 5, 6), (2, 2, 2), 0.0, 2, dict(yield_stress=2e3, viscosity=5.0)),
    ((9, 5, 6), (2, 2, 2), 0.1, 2, dict(mass=0.05)),
])
def test_few_and_many_bricks_agree_bitwise(pkg, cells, k, jitter, codes, kw):
    rng = np.random.default_rng(3)
    X = _lattice(cells, k) + jitter * DX / 2 * rng.uniform(-1, 1, (np.prod(cells) * np.prod(k), 3))
    X = X.astype(np.float32).astype(np.float64)
    sc, n = _scene(X, codes < 12, **kw), len(X)
    q = np.floor(X / DX).astype(int)
    # slabs along x, or for twelve codes columns; 0: none, odd / even: side 1 / 2 of a cut
    code = q[:, 0] * codes // cells[0] if codes < 12 else q[:, 0] % 4 + 4 * (q[:, 1] % 3)
    cut = 1 + (code + 1) // 2
    state = dict(v=(0.3 * rng.standard_normal((n, 3))).astype(np.float32),
                 F=(np.eye(3).ravel() + 0.02 * rng.standard_normal((n, 9))).astype(np.float32),
                 mask1=np.where(code % 2 == 1, 1 << cut, 0).astype(np.uint32),
                 mask2=np.where((code % 2 == 0) & (code > 0), 1 << cut, 0).astype(np.uint32))
    filler = _scene(_lattice((42, 42, 42), (1, 1, 1)), False)   # over 1,000 bricks and 608 node tiles
    got = []
    for many in (False, True):
        s = pkg.Scene(sc)
        s.write(**state)
        if many:
            specs = [sc, filler]
            fp = [pkg.footprint(q) for q in specs]
            b = pkg.Batch(max_particles=sum(q.n for q in specs), max_nodes=sum(f[1] for f in fp),
                          max_scenes=2, max_bricks=sum(f[2] for f in fp))
            assert fp[1][2] > 4 * 152 and fp[1][1] > 4 * 152 * 128
            f = pkg.Scene(filler)
            b.add(f)
            b.add(s)
            b.step(8)
        else:
            assert pkg.footprint(sc)[2] <= 2 * 152
            s.step(8)
        got.append((s.read(*FIELDS), s.tool_wrench() if codes < 12 else 0, s.info().error_bits, s.info().n_slots,
                    s.tool_state() if codes < 12 else np.zeros(1)))
        s.close()
        if many:
            f.close()
            b.close()
    for name in FIELDS:
        assert np.array_equal(got[0][0][name], got[1][0][name]), name
    assert np.array_equal(got[0][1], got[1][1]) and got[0][2:4] == got[1][2:4]
    assert np.array_equal(got[0][4], got[1][4])
    assert got[0][2] == 0
    if codes < 12 and n > 1:
        assert np.any(got[0][1] != 0)
