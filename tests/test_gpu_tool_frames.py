"""The frame that a set tool state sets up is the one that stepping would have
left: setting a tool to the state it is in changes no bit of what follows."""
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


def _scene(mass, tilt):
    X = bi.lattice_cuboid((0.04, 0.02, 0.02), DX)
    edge = (X[:, 0].mean() + 2e-4, X[:, 1].mean(), X[:, 2].max() - 0.2 * DX)
    c, s = np.cos(tilt), np.sin(tilt)
    R = np.array([[c, -s, 0], [s, c, 0], [0, 0, 1.0]]) @ np.array([[1, 0, 0], [0, c, -s], [0, s, c]])
    b = bi.Blade(pose_x=tuple(float(t) for t in edge), pose_R=tuple(R.ravel()), edge_point=(1e-4, -2e-4, 3e-4), mass=mass,
                 inertia=tuple((4e-5 * mass * np.array([[1, .1, .2], [.1, 2, .3], [.2, .3, 3]])).ravel()),
                 segments=[bi.Segment(9, v=(0.1, 0.0, -1.5), omega=(0.5, 2.0, -1.0), cut_id=0),
                           bi.Segment(40, v=(0.0, 0.2, -1.5), omega=(-1.0, 0.3, 2.0), cut_id=1)])
    return bi.Scene(X=X, dx=DX, V0=DX ** 3 / 8, dt=1e-4, blade=b)


@pytest.mark.parametrize("mass", [0.0, 0.05])
@pytest.mark.parametrize("batched", [False, True])
def test_setting_the_tool_where_it_is_changes_nothing(pkg, mass, batched):
    specs = [_scene(mass, t) for t in (0.1, -0.7, 0.4)]
    fp = [pkg.footprint(q) for q in specs]
    got = []
    for touch in (False, True):
        if batched:
            b = pkg.Batch(max_particles=sum(f[0] for f in fp), max_nodes=sum(f[1] for f in fp), max_scenes=3,
                          max_bricks=sum(f[2] for f in fp))
            ss = [pkg.Scene.in_batch(b, q) for q in specs]
        else:
            ss = [pkg.Scene(q) for q in specs]
        for _ in range(6):      # 3 substeps at a time, over the change of cuts
            if touch and batched:
                b.set_tool_states(np.stack([s.tool_state() for s in ss]))
            elif touch:
                for s in ss:
                    t = s.tool_state()
                    s.set_tool_state(t[:3], t[3:12], t[12:15], t[15:])
            if batched:
                b.step(3)
            else:
                for s in ss:
                    s.step(3)
        got.append([(s.read(*FIELDS), s.tool_state(), s.tool_wrench(), s.info().error_bits) for s in ss])
        for s in ss:
            s.close()
        if batched:
            b.close()
    for a, c in zip(*got):
        for k in FIELDS:
            assert np.array_equal(a[0][k], c[0][k]), k
        assert np.array_equal(a[1], c[1]) and np.array_equal(a[2], c[2]) and a[3] == c[3] == 0
        assert np.any(a[2] != 0)
