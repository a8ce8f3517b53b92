"""Lattice brick kernels against the general ones, bit for bit.

A body whose particles lie on planes of at most two per base cell takes the
lattice kernels.  The same body plus three far-away particles that share a
base cell on three planes takes the general kernels; the three touch none of
its nodes, so every particle of the body must come out with the same bits.
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


def _planes(cells, offsets):
    """Tensor grid: the offsets (in cells) of each axis's planes in every cell."""
    ax = [(np.arange(n)[:, None] + np.asarray(o)[None, :]).ravel() * DX for n, o in zip(cells, offsets)]
    return np.stack(np.meshgrid(*ax, indexing="ij"), -1).reshape(-1, 3)


TWO, ONE = (0.25, 0.75), (0.5,)


def _body(name):
    rng = np.random.default_rng(5)
    if name == "aligned":           # full bricks and ragged ends
        return _planes((9, 5, 6), (TWO,) * 3), -DX / 2
    if name == "unaligned":         # base cells hold parts of two lattice cells
        return _planes((9, 5, 6), (TWO,) * 3), 0.0
    if name == "one_per_cell":
        return _planes((7, 4, 5), (ONE,) * 3), -DX / 2
    if name == "mixed_planes":      # 2 x 1 x 2 per cell
        return _planes((7, 4, 5), (TWO, ONE, TWO)), 0.0
    if name == "uneven_planes":     # planes not evenly spaced
        return _planes((6, 5, 5), ((0.2, 0.71), (0.37, 0.9), (0.11, 0.5))), -DX / 2
    if name == "holes":
        X = _planes((9, 5, 6), (TWO,) * 3)
        return X[rng.random(len(X)) < 0.6], -DX / 2
    if name == "single":
        return np.array([[0.5, 0.5, 0.5]]) * DX, 0.0
    if name == "one_brick":
        return _planes((4, 4, 4), (TWO,) * 3), -DX / 2
    raise KeyError(name)


def _codes(kind, X, rng):
    """Side masks of cuts 1 and up (cut 0 is the blade's own)."""
    n = len(X)
    code = np.zeros(n, int)      # 0: none; odd / even: digit 1 / 2 of a cut
    if kind == "cut":            # an oblique cut through the middle, most of the body unlabelled
        s = (X - X.mean(0)) @ np.array([1.0, 0.3, 0.1])
        code = np.where(np.abs(s) < 1.5 * DX, np.where(s < 0, 1, 2), 0)
    elif kind == "random3":      # three codes in no spatial order: every node holds all of them
        code = rng.integers(0, 3, n)
    elif kind == "columns12":    # twelve codes, a column of cells each
        q = np.floor((X - X.min(0)) / DX + 1e-6).astype(int)
        code = q[:, 0] % 4 + 4 * (q[:, 1] % 3)
    cut = 1 + (code + 1) // 2
    return (np.where(code % 2 == 1, 1 << cut, 0).astype(np.uint32),
            np.where((code % 2 == 0) & (code > 0), 1 << cut, 0).astype(np.uint32))


def _scene(X, origin, cut_id=0, **kw):
    size = X.max(0) - X.min(0) + DX
    # the edge reaches the top particles' centres (labels) after ten substeps
    edge = (X[:, 0].mean() + 2e-4, X[:, 1].mean(), X[:, 2].max() + 0.25 * DX)
    blade = bi.Blade(pose_x=tuple(float(t) for t in edge), half_length=float(size.max()),
                     segments=[bi.Segment(40, v=(0.0, 0.0, -1.5), cut_id=cut_id)])
    return bi.Scene(X=X, dx=DX, origin=(origin,) * 3, V0=DX ** 3 / 8, dt=1e-4, E=1e5, nu=0.3, blade=blade, **kw)


# random3 and columns12 in one brick: more tile slots than the general kernel's
# shared-memory window (the blade adds no labels there, the slot pool is full);
# columns12 has more codes than the lattice kernels' slot table
@pytest.mark.parametrize("body,codes,kw", [
    ("aligned", "none", {}), ("aligned", "cut", {}), ("unaligned", "cut", {}),
    ("one_per_cell", "cut", {}), ("mixed_planes", "none", {}), ("uneven_planes", "cut", {}),
    ("holes", "cut", {}), ("single", "none", {}), ("one_brick", "random3", dict(cut_id=-1)),
    ("one_brick", "columns12", dict(cut_id=-1)),
    ("aligned", "cut", dict(model="fixed_corotated", yield_stress=2e3, viscosity=5.0)),
    ("unaligned", "cut", dict(pair_contact=True)),
])
def test_lattice_kernels_equal_the_general_ones_bitwise(pkg, body, codes, kw):
    X, origin = _body(body)
    X = X.astype(np.float32).astype(np.float64)
    rng = np.random.default_rng(7)
    n = len(X)
    far = X.max(0)[None, :] + np.array([[12.1, 0.0, 0.0], [12.2, 0.1, 0.1], [12.3, 0.2, 0.2]]) * DX
    far = np.floor(far / DX) * DX + np.array([[0.6, 0.6, 0.6], [0.7, 0.7, 0.7], [0.8, 0.8, 0.8]]) * DX
    m1, m2 = _codes(codes, X, rng)
    state = dict(v=(0.3 * rng.standard_normal((n, 3))).astype(np.float32),
                 F=(np.eye(3).ravel() + 0.02 * rng.standard_normal((n, 9))).astype(np.float32), mask1=m1, mask2=m2)
    got = []
    for extra in (0, 3):
        sc = _scene(X, origin, **kw).replace(X=np.concatenate([X, far[:extra]]))
        pad = {"v": np.zeros((extra, 3)), "F": np.tile(np.eye(3).ravel(), (extra, 1)),
               "mask1": np.zeros(extra), "mask2": np.zeros(extra)}
        g = pkg.Scene(sc, wrench_history=20)
        g.write(**{k: np.concatenate([a, pad[k].astype(a.dtype)]) for k, a in state.items()})
        g.step(20)
        r = {k: a[:n] for k, a in g.read(*FIELDS).items()}
        r["wrench"] = g.wrench_history(0, 20)
        assert g.info().error_bits == 0
        got.append(r)
        g.close()
    for k in got[0]:
        assert np.array_equal(got[0][k], got[1][k]), k
    assert np.any(got[0]["x"] != X.astype(np.float32))
