"""Timed workloads of the TLMPM cutting library, through its public calls.

Every case starts from a body in the middle of a cut: material behind the
blade's edge carries its side labels and stands clear of the blade, the body
moves and is strained by smooth seeded fields, and the blade advances.  Sizes
and materials are those of the repository's workloads: cuboids of 4k to 64k
particles in batches, single bodies up to 500k, the 0.2 m cylinder with two
intersecting cuts, and the 16-per-cell calibration cuboid.

Kinds of pass:
  tick         set the tool, advance one control interval, read wrench and state
  rollout      restore a checkpoint, advance, read the result (a planner's sample)
  batch        advance many scenes by CUDA-graph launches, read all of them
  contact      rollout with material-material contact and a two-way tool
  surface      rebuild and embed the displayed surface, copy it out
  calibration  loss and gradient of a force trajectory (forward and backward)

Reaction wrenches and gradients are sums of 32-bit particle impulses that the
calls hand over in doubles; a pass returns them at their 32-bit precision.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2609_27342_gb300 as bm
from paper_2609_27342_gb300 import calibration, sim, surface

RHO = 1000.0
STATE_BYTES = 156.0     # state one substep must read and write, per particle
STEP_FLOPS = 500.0      # contact, stress and separable transfers, per particle


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # a 1 kHz control loop on a small body: latency and launches count
        dict(name="tick_4k", kind="tick", cells="12x6x7", lattice="2x2x2", aligned=False, jitter=0.0,
             substeps=10, E=1e5, nu=0.3, dx=5e-3, cuts=1, material="elastic"),
        # the single-cut cuboid as one sample of a sampling planner
        dict(name="rollout_16k", kind="rollout", cells="20x10x10", lattice="2x2x2", aligned=False, jitter=0.0,
             substeps=10, E=1e5, nu=0.3, dx=5e-3, cuts=1, material="elastic"),
        # an odd-sized plastic, viscous body sampled off the lattice (a scan)
        dict(name="rollout_scan_21k", kind="rollout", cells="17x13x12", lattice="2x2x2", aligned=True, jitter=0.2,
             substeps=10, E=1e5, nu=0.35, dx=5e-3, cuts=2, material="plastic"),
        # the benchmark: 256 uneven scenes in one graph launch
        dict(name="batch_256", kind="batch", scenes=256, n_min=4096, n_max=65536, sizes_seed=2, substeps=20,
             dx=5e-3, cuts=1),
        # one served rollout at the upper end of the request sizes, third cut
        dict(name="large_477k", kind="batch", scenes=1, n_min=500000, n_max=500000, sizes_seed=3, substeps=20,
             dx=5e-3, cuts=3),
        # two intersecting cuts, two-way tool, faces touching: the contact path
        dict(name="contact_cylinder", kind="contact", length=100, radius=10, substeps=10, E=5e4, nu=0.35, dx=2e-3,
             cuts=2),
        # one displayed frame of the same body
        dict(name="surface_cylinder", kind="surface", length=100, radius=10, E=5e4, nu=0.35, dx=2e-3, cuts=2,
             planes_seed=4),
        # one optimiser step of the material calibration, shortened horizon
        dict(name="calibration_32k", kind="calibration", cells="20x10x10", lattice="4x2x2", substeps=30, every=10,
             E=1e5, nu=0.3, dx=5e-3),
    ]


def draw(rng):
    kind = rng.choice(["tick", "rollout", "rollout", "batch", "batch", "contact", "surface", "calibration"])

    def log(a, b):
        return math.exp(rng.uniform(math.log(a), math.log(b)))

    def cells(n):
        ny = max(2, round((n / 16.0) ** (1 / 3)))
        nx = max(2, round(n / 8.0 / ny / ny * rng.uniform(0.8, 1.2)))
        return "%dx%dx%d" % (nx, ny + rng.randint(0, 1), ny)

    nu = round(rng.uniform(0.25, 0.45), 3)
    if kind in ("tick", "rollout"):
        return dict(kind=kind, cells=cells(log(4096, 65536)), lattice="2x2x2", aligned=rng.random() < 0.5,
                    jitter=rng.choice([0.0, 0.0, 0.2]), substeps=rng.randint(5, 10),
                    E=round(log(2e4, 2e5)), nu=nu, dx=5e-3, cuts=rng.randint(1, 2),
                    material=rng.choice(["elastic", "elastic", "corotated", "plastic"]))
    if kind == "batch":
        return dict(kind=kind, scenes=round(log(2, 128)), n_min=4096, n_max=65536,
                    sizes_seed=rng.randint(10, 10 ** 6), substeps=rng.randint(8, 20), dx=5e-3, cuts=rng.randint(1, 2))
    if kind in ("contact", "surface"):
        c = dict(kind=kind, length=rng.randint(30, 100), radius=rng.randint(5, 10), E=round(log(2e4, 1e5)), nu=nu,
                 dx=2e-3, cuts=rng.randint(1, 2))
        return dict(c, substeps=rng.randint(5, 10)) if kind == "contact" else dict(c, planes_seed=rng.randint(10, 10 ** 6))
    return dict(kind=kind, cells=cells(log(4096, 16384)), lattice=rng.choice(["4x2x2", "2x2x2"]),
                substeps=rng.randint(15, 30), every=rng.randint(7, 15), E=round(log(5e4, 2e5)), nu=nu, dx=5e-3)


# ---------------------------------------------------------------------------
# scenes and states
# ---------------------------------------------------------------------------
def _ints(text):
    return [int(t) for t in text.split("x")]


def _lattice(cells, k, dx):
    ax = [((np.arange(n * q) + 0.5) / q) * dx for n, q in zip(cells, k)]
    return np.stack(np.meshgrid(*ax, indexing="ij"), -1).reshape(-1, 3)


def _plane(rng, tilt):
    """Blade axes (normal, edge, front): front downwards, normal turned about z, tilted."""
    a = rng.uniform(-0.4, 0.4)
    n = np.array([math.cos(a), math.sin(a), math.tan(tilt)])
    n /= np.linalg.norm(n)
    d = np.array([0.0, 0.0, -1.0])
    d -= d.dot(n) * n
    d /= np.linalg.norm(d)
    return n, np.cross(d, n), d


def _scene(rng, X, size, case, E, nu, per_cell, origin, speed, n_cuts, pair=False, planes=None):
    """A scene description and its mid-cut state (x, v, F, side masks); `planes` places the cuts."""
    planes = planes or rng
    dx = case["dx"]
    V0 = dx ** 3 / per_cell
    lam, mu = E * nu / ((1 + nu) * (1 - 2 * nu)), E / (2 * (1 + nu))
    dt = min(5e-5 if pair else 1e-4, 0.3 * dx / math.sqrt((lam + 2 * mu) / RHO))
    X = np.asarray(X, np.float32)
    n, e, d = _plane(planes, planes.uniform(-0.3, 0.3))
    centre = np.asarray(size) / 2
    edge = centre + n * planes.uniform(-0.25, 0.25) * dx
    half_thick, Rp = 5e-4, V0 ** (1 / 3) / 2
    long_edge = 0.05 if pair else float(max(size))
    mass, inertia = 0.0, (0.0,) * 9
    if pair:
        mass = 0.2
        a, b, c = 2 * half_thick, 2 * long_edge, 0.1
        inertia = (mass * (b * b + c * c) / 12, 0.0, 0.0, 0.0, mass * (a * a + c * c) / 12, 0.0, 0.0, 0.0,
                   mass * (a * a + b * b) / 12)
    blade = SimpleNamespace(
        edge_point=(0.0, 0.0, 0.0), normal=(1.0, 0.0, 0.0), edge_dir=(0.0, 1.0, 0.0), front_dir=(0.0, 0.0, 1.0),
        half_length=long_edge, thickness=2 * half_thick, height=0.1, mu_s=0.2, mu_d=0.2, mass=mass, inertia=inertia,
        pose_x=tuple(edge), pose_R=tuple(np.stack([n, e, d], 1).ravel()), servo_gain=0.0, rigid_interval=1,
        segments=[SimpleNamespace(n_steps=1000000, v=tuple(speed * d), omega=(0.0, 0.0, 0.0), cut_id=n_cuts - 1)])
    material = case.get("material", "elastic")
    spec = SimpleNamespace(
        X=X, E=E, nu=nu, rho=RHO, dx=dx, origin=origin, V0=V0, dt=dt, beta=0.99, gravity=(0.0, 0.0, -9.81),
        floor=True, floor_z=0.0, s_R=1.0, s_n=1.0, gamma_k=0.5, gamma_c=0.5, pair_contact=pair, pair_mu_s=0.2,
        pair_mu_d=0.2, G_c=50.0, zeta=0.9, u_min=1e-3, b_back=-1.0, b_lead=-1.0, band_half_width=-1.0,
        tool_contact=True, blade=blade, model="neo_hookean" if material == "elastic" else "fixed_corotated",
        yield_stress=2e3 if material == "plastic" else 0.0, viscosity=5.0 if material == "plastic" else 0.0)
    # labels: earlier cuts went right through, on planes of their own; the
    # current cut reaches down to the edge
    N = len(X)
    m1, m2 = np.zeros(N, np.uint32), np.zeros(N, np.uint32)
    x = X.astype(np.float64)
    for k in range(n_cuts - 1):
        q, _, _ = _plane(planes, 0.0)
        # stacked along the body; in the cylinder the two cuts intersect
        s = (x - centre) @ q - ((2 * k - 1) * 0.3 if case["kind"] in ("batch", "tick", "rollout") else 0.01) * size[0]
        band = np.abs(s) <= 6 * dx
        m1[band & (s < 0)] |= np.uint32(1 << k)
        m2[band & (s >= 0)] |= np.uint32(1 << k)
    r = x - edge
    s, f = r @ n, r @ d
    band = (np.abs(s) <= 6 * dx) & (f <= 0) & (f >= -0.1)
    m1[band & (s < 0)] |= np.uint32(1 << (n_cuts - 1))
    m2[band & (s >= 0)] |= np.uint32(1 << (n_cuts - 1))
    # positions: the faces and the material under the edge rest against the blade
    clear = half_thick + Rp
    side = (f <= 0) & (np.abs(s) < clear)
    s_new = np.where(side, np.where(s < 0, -1.0, 1.0) * (clear + 0.2 * np.abs(s) - 1e-6 * rng.random(N)), s)
    reach = np.sqrt(np.maximum(Rp ** 2 - np.maximum(np.abs(s) - half_thick, 0.0) ** 2, 0.0))
    under = (f > 0) & (f < reach)
    f_new = np.where(under, reach - 1e-6 * rng.random(N), f)
    x += (s_new - s)[:, None] * n + (f_new - f)[:, None] * d
    # smooth motion and strain of the body, and fine noise
    u = (X - centre.astype(np.float32)) / np.float32(max(size))

    def wave(lo, hi, width):
        k, phase = rng.uniform(lo, hi, (3, width)), rng.uniform(0, 6, width)
        return np.sin(u @ k.astype(np.float32) + phase.astype(np.float32))

    v = np.float32(0.2) * wave(1.0, 3.0, 3) + rng.uniform(-0.2, 0.2, 3).astype(np.float32)
    v += np.float32(0.01) * rng.standard_normal((N, 3), dtype=np.float32)
    F = np.float32(0.01) * wave(-3.0, 3.0, 9)
    F += np.float32(1e-3) * rng.standard_normal((N, 9), dtype=np.float32)
    F += np.eye(3, dtype=np.float32).ravel()
    return spec, dict(x=x.astype(np.float32), v=v.astype(np.float32), F=F, mask1=m1, mask2=m2)


def _single(case, rng):
    cells, k = _ints(case["cells"]), _ints(case["lattice"])
    dx = case["dx"]
    size = np.array(cells) * dx
    X = _lattice(cells, k, dx)
    if case.get("jitter", 0.0):
        X += rng.uniform(-case["jitter"], case["jitter"], X.shape) * (dx / np.array(k))
    o = -dx / 2 if case.get("aligned", False) else 0.0
    return _scene(rng, X, size, case, float(case["E"]), case["nu"], math.prod(k), (o,) * 3, 0.2,
                  case.get("cuts", 1))


def _batch(case, rng):
    layout = np.random.default_rng(case["sizes_seed"])   # sizes and materials belong to the case
    out = []
    for _ in range(case["scenes"]):
        dx = case["dx"]
        N = math.exp(layout.uniform(math.log(case["n_min"]), math.log(case["n_max"])))
        ny = max(2, round((N / 16.0) ** (1 / 3)))
        E, nu = math.exp(layout.uniform(math.log(1e4), math.log(1e6))), layout.uniform(0.25, 0.45)
        cells = (2 * ny, ny, ny)
        out.append(_scene(rng, _lattice(cells, (2, 2, 2), dx), np.array(cells) * dx, case, E, nu, 8,
                          (-dx / 2,) * 3, layout.uniform(0.05, 0.5), case["cuts"]))
    return out


def _cylinder(case, rng, pair):
    dx, R = case["dx"], case["radius"] * case["dx"]
    cells = (case["length"], 2 * case["radius"], 2 * case["radius"])
    X = _lattice(cells, (2, 2, 2), dx)
    X = X[(X[:, 1] - R) ** 2 + (X[:, 2] - R) ** 2 <= R * R]
    return _scene(rng, X, np.array(cells) * dx, case, float(case["E"]), case["nu"], 8, (0.0,) * 3, 1.0,
                  case["cuts"], pair=pair, planes=None if pair else np.random.default_rng(case["planes_seed"]))


def _buffers(n, names):
    width = {"x": 3, "v": 3, "F": 9}
    return {k: torch.empty((n, width[k]), dtype=torch.float32, device="cuda") if k in width
            else torch.empty(n, dtype=torch.int32, device="cuda") for k in names}


def _wrench(w):
    return torch.from_numpy(w).to(torch.float32)


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    st = SimpleNamespace(kind=kind, case=case)
    if kind == "calibration":
        spec, _ = _single(dict(case, aligned=False), rng)
        # from rest, the edge just above the top; a measured force trajectory
        size, b, n = np.array(_ints(case["cells"])) * case["dx"], spec.blade, case["substeps"]
        b.pose_x = (size[0] / 2 + rng.uniform(-1e-3, 1e-3), size[1] / 2,
                    float(spec.X[:, 2].max()) + spec.V0 ** (1 / 3) / 2 + 5e-5 * rng.random())
        b.pose_R = (1.0, 0.0, 0.0, 0.0, -1.0, 0.0, 0.0, 0.0, -1.0)
        b.segments[0].v = (0.0, 0.0, -0.2)
        st.spec = spec
        st.target = np.array([[0.02, 0.02, 0.5]]) * np.linspace(0, 1, n)[:, None] + 0.01 * rng.standard_normal((n, 3))
        return st
    if kind == "batch":
        specs = _batch(case, rng)
        fp = [sim.footprint(s) for s, _ in specs]
        st.batch = bm.Batch(max_particles=sum(f[0] for f in fp), max_nodes=sum(f[1] for f in fp),
                            max_scenes=len(fp), max_bricks=sum(f[2] for f in fp))
        st.scenes = []
        for spec, state in specs:
            s = bm.Scene.in_batch(st.batch, spec)
            s.write(**state)
            st.scenes.append(s)
        st.out = _buffers(sum(s.n for s in st.scenes), ["x", "F"])
        first = np.cumsum([0] + [s.n for s in st.scenes])
        st.views = [{k: t[a:b] for k, t in st.out.items()} for a, b in zip(first, first[1:])]
        return st
    spec, state = _single(case, rng) if kind in ("tick", "rollout") else _cylinder(case, rng, kind == "contact")
    st.scene = bm.Scene(spec)
    st.scene.write(**state)
    if kind == "surface":
        st.scene.step(1)    # the cut in progress records its plane
        x = st.scene.read("x")["x"]
        st.scene.write(x=x + np.float32(1e-3) * np.sin(x @ rng.uniform(-60.0, 60.0, (3, 3)).astype(np.float32)))
        st.surface = surface.Surface(st.scene, (2, 2, 2))
        return st
    st.out = _buffers(st.scene.n, ["x", "F", "mask1", "mask2"] + ([] if kind == "contact" else ["v"]))
    if kind == "tick":
        st.tool = (spec.blade.pose_x, spec.blade.pose_R, spec.blade.segments[0].v, (0.0, 0.0, 0.0))
    else:
        st.checkpoint = st.scene.checkpoint()
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(st):
    if st.kind == "calibration":
        loss, g = calibration.force_loss_and_grad(st.spec, st.target, st.case["substeps"], st.case["every"])
        theta = np.concatenate([[g["E"], g["nu"]], np.ravel(g["v_seg"])])
        return {"loss": torch.tensor(loss, dtype=torch.float32), "gradient": torch.from_numpy(theta).float(),
                "forces": torch.from_numpy(g["forces"]).float()}
    if st.kind == "surface":
        nv, nt = st.surface.update(rebuild=True)
        vertices = torch.empty((nv, 3), dtype=torch.float32, device="cuda")
        triangles = torch.empty((nt, 3), dtype=torch.int32, device="cuda")
        st.surface.read_into(vertices, triangles)
        return {"vertices": vertices, "triangles": triangles}
    if st.kind == "batch":
        st.batch.step(st.case["substeps"])
        wrench = _wrench(st.batch.tool_wrenches())
        for s, view in zip(st.scenes, st.views):
            s.read_device(view)
        return dict(st.out, wrench=wrench)
    if st.kind == "tick":
        st.scene.set_tool_state(*st.tool)
    else:
        st.scene.restore(st.checkpoint)
    st.scene.step(st.case["substeps"])
    wrench = _wrench(st.scene.tool_wrench())
    st.scene.read_device(st.out)
    return dict(st.out, wrench=wrench)


def _particles(case):
    if case["kind"] == "batch":
        layout = np.random.default_rng(case["sizes_seed"])
        total = 0
        for _ in range(case["scenes"]):
            N = math.exp(layout.uniform(math.log(case["n_min"]), math.log(case["n_max"])))
            layout.uniform(size=3)
            total += 16 * max(2, round((N / 16.0) ** (1 / 3))) ** 3
        return total
    if case["kind"] in ("contact", "surface"):
        return 8 * case["length"] * math.pi * case["radius"] ** 2
    return math.prod(_ints(case["cells"])) * math.prod(_ints(case["lattice"]))


def work(case):
    n = _particles(case)
    if case["kind"] == "surface":
        # lattice codes, positions and reference positions in; about one
        # vertex per boundary lattice point, two triangles each, out
        verts = 4 * case["length"] * 2 * math.pi * case["radius"] * 1.3
        return {"bytes": n * 32.0 + verts * 36.0, "flops": verts * 2000.0}
    steps = case["substeps"]
    if case["kind"] == "calibration":   # forward, recomputation and adjoint
        return {"bytes": n * steps * (2 * STATE_BYTES + 320.0), "flops": n * steps * (2 * STEP_FLOPS + 1000.0)}
    per = STATE_BYTES + (100.0 if case["kind"] == "contact" else 0.0)
    return {"bytes": n * (steps * per + 96.0), "flops": n * steps * STEP_FLOPS}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------
def _spline(f):
    a, b, c = 1.5 - f, f - 1.0, f - 0.5
    return torch.stack([0.5 * a * a, 0.75 - b * b, 0.5 * c * c], -1), torch.stack([-a, -2 * b, c], -1)


def _cofactor(F):
    a, b, c = F[:, 0], F[:, 1], F[:, 2]
    return torch.stack([torch.linalg.cross(b, c), torch.linalg.cross(c, a), torch.linalg.cross(a, b)], 1)


def _elastic(F, spec, mu, lam):
    cof = _cofactor(F)
    J = (F[:, 0] * cof[:, 0]).sum(-1)[:, None, None]
    if spec.model == "neo_hookean":
        inv = cof / J
        return mu * (F - inv) + lam * torch.log(J) * inv
    U, _, Vh = torch.linalg.svd(F)
    return 2 * mu * (F - U @ Vh) + lam * (J - 1) * cof


def _stress(F, Fpi, Fdot, spec, mu, lam):
    """First Piola stress (fixed-corotated or neo-Hookean, von Mises, Newtonian viscosity); updates Fpi."""
    if spec.yield_stress > 0:
        Fe = F @ Fpi
        U, S, Vh = torch.linalg.svd(Fe)
        h = torch.log(S)
        mean = h.mean(-1, keepdim=True)
        dev = h - mean
        q = math.sqrt(6.0) * mu * dev.norm(dim=-1, keepdim=True)
        scale = torch.where(q > spec.yield_stress, spec.yield_stress / q.clamp_min(1e-300), torch.ones_like(q))
        Fe = torch.where((q > spec.yield_stress)[:, :, None], U @ torch.diag_embed(torch.exp(mean + scale * dev)) @ Vh,
                         Fe)
        Fpi.copy_(torch.linalg.solve(F, Fe))
        P = _elastic(Fe, spec, mu, lam) @ Fpi.mT
    else:
        P = _elastic(F, spec, mu, lam)
    if spec.viscosity > 0:
        L = Fdot @ torch.linalg.inv(F)
        P = P + spec.viscosity * (L + L.mT) @ _cofactor(F)
    return P


def _blade_contact(x, v, m, spec, tool, hist, D, cut, reset):
    """Impulse on each particle, reaction wrench, new friction history and cutting progress."""
    b, dt = spec.blade, spec.dt
    xB, ax, vB = tool["x"], tool["R"].T, tool["v"]
    Rp, hx = spec.s_R * spec.V0 ** (1 / 3) / 2, torch.tensor([b.thickness / 2, b.half_length, b.height / 2]).to(x)
    centre = xB - hx[2] * ax[2]
    q = (x - centre) @ ax.T
    out = (q.abs() > hx).any(-1)
    qc = q.clamp(-hx, hx)
    dist = (q - qc).norm(dim=-1)
    inner = hx - q.abs()
    best = torch.nn.functional.one_hot(inner.argmin(-1), 3).to(x)
    sign = torch.where(q < 0, -1.0, 1.0) * best
    nl = torch.where(out[:, None], (q - qc) / dist.clamp_min(1e-300)[:, None], sign)
    phi = torch.where(out, dist, -inner.min(-1).values) - Rp
    xc = centre + torch.where(out[:, None], qc, torch.where(best > 0, sign * hx, q)) @ ax
    nB = nl @ ax
    vrel = v - vB
    vn = (vrel * nB).sum(-1)
    gap = phi + dt * vn.clamp_max(0.0)
    Jn = spec.s_n * m / dt * (-gap).clamp_min(0.0)
    tu = hist - (hist * nB).sum(-1, keepdim=True) * nB
    tl = tu.norm(dim=-1, keepdim=True)
    ut = torch.where(tl > 0, tu * hist.norm(dim=-1, keepdim=True) / tl.clamp_min(1e-300), torch.zeros_like(tu))
    vt = vrel - vn[:, None] * nB
    kt = spec.gamma_k * m / dt ** 2
    ct = 2 * spec.gamma_c * math.sqrt(m * kt)
    trial = -kt * ut - ct * vt
    fl, lim = trial.norm(dim=-1, keepdim=True), (Jn / dt)[:, None]
    stick = fl <= b.mu_s * lim
    ft = torch.where(stick, trial, b.mu_d * lim / fl.clamp_min(1e-300) * trial)
    new = torch.where(stick, ut + dt * vt, -(ft + ct * vt) / kt)
    on = (Jn > 0)[:, None]
    JB = torch.where(on, Jn[:, None] * nB + dt * ft, torch.zeros_like(ft))
    r = x - xB
    s, l, f = r @ ax[0], r @ ax[1], r @ ax[2]
    uc = (vB - v) @ ax[2]
    h, back, lead = 6 * spec.dx, spec.dx, spec.dx
    D = torch.zeros_like(D) if reset else D
    front = on[:, 0] & (s.abs() <= h) & (l.abs() <= b.half_length) & (f >= 0) & (f <= lead) & (uc > spec.u_min)
    Jc = (JB @ ax[2]).clamp_min(0.0)
    free = front & (D >= 1)
    W = spec.G_c * spec.V0 ** (2 / 3) * (1 - spec.zeta) / spec.zeta
    D = torch.where(front & (D < 1), (D + Jc * uc / W).clamp_max(1.0), D)
    JB = JB - torch.where(free, Jc, torch.zeros_like(Jc))[:, None] * ax[2]
    FB = -JB / dt
    wrench = torch.cat([FB.sum(0), torch.linalg.cross(xc - xB, FB).sum(0)])
    band = (s.abs() <= h) & (l.abs() <= b.half_length) & (f <= 0) & (f >= -back - (uc * dt).clamp_min(0.0))
    label = torch.where(band, torch.where(s < 0, 1, 2), 0)
    return JB, wrench, torch.where(on, new, torch.zeros_like(new)), D, label


def _couple(S, mass, codes):
    """Coupling of the compatible logical grids: S (codes, nodes, c), mass (codes, nodes)."""
    M = mass.sum(0).clamp_min(1e-300)[:, None]
    out = S.clone()
    for a, (a1, a2) in enumerate(codes):
        for b, (b1, b2) in enumerate(codes):
            if a != b and not (a1 & b2) | (a2 & b1):
                out[a] += (mass[a][:, None] * S[b] - mass[b][:, None] * S[a]) / M
    return out


def _rollout64(spec, state, steps):
    dev = "cuda"
    t = lambda a: torch.as_tensor(np.asarray(a), dtype=torch.float64, device=dev)  # noqa: E731
    X, x, v, F = t(spec.X), t(state["x"]), t(state["v"]), t(state["F"]).reshape(-1, 3, 3)
    m1, m2 = (torch.as_tensor(state[k].astype(np.int64), device=dev) for k in ("mask1", "mask2"))
    N, dt, dx = len(X), spec.dt, spec.dx
    m = spec.rho * spec.V0
    lam, mu = spec.E * spec.nu / ((1 + spec.nu) * (1 - 2 * spec.nu)), spec.E / (2 * (1 + spec.nu))
    g = t(spec.gravity)
    grid = (X - t(spec.origin)) / dx
    base = torch.floor(grid - 0.5)
    w, dw = _spline(grid - base)
    base = (base - base.min(0).values).long()
    dims = (base.max(0).values + 3).tolist()
    n_nodes = math.prod(dims)
    idx, Ns, gN = [], [], []
    for i in range(3):
        for j in range(3):
            for k in range(3):
                idx.append(((base[:, 0] + i) * dims[1] + base[:, 1] + j) * dims[2] + base[:, 2] + k)
                Ns.append(w[:, 0, i] * w[:, 1, j] * w[:, 2, k])
                gN.append(torch.stack([dw[:, 0, i] * w[:, 1, j] * w[:, 2, k], w[:, 0, i] * dw[:, 1, j] * w[:, 2, k],
                                       w[:, 0, i] * w[:, 1, j] * dw[:, 2, k]], -1) / dx)
    b = spec.blade
    tool = dict(x=t(b.pose_x), R=t(b.pose_R).reshape(3, 3), v=t(b.segments[0].v))
    cut, hist, D = b.segments[0].cut_id, torch.zeros_like(x), torch.zeros(N, dtype=torch.float64, device=dev)
    Fpi, Fdot = torch.eye(3, dtype=torch.float64, device=dev).repeat(N, 1, 1), torch.zeros_like(F)
    wrench, forces = None, []
    for step in range(steps):
        pairs, cid = torch.unique(torch.stack([m1, m2], 1), dim=0, return_inverse=True)
        codes = [tuple(p) for p in pairs.tolist()]
        rows = [cid * n_nodes + q for q in idx]
        total = len(codes) * n_nodes

        def scatter(parts, width):
            S = torch.zeros((total, width), dtype=torch.float64, device=dev)
            for q, val in zip(rows, parts):
                S.index_add_(0, q, val)
            return S.reshape(len(codes), n_nodes, width)

        JB, wrench, hist, D, label = _blade_contact(x, v, m, spec, tool, hist, D, cut, step == 0)
        forces.append(wrench[:3])
        J = JB + m * g * dt
        gap = x[:, 2] - spec.floor_z - spec.s_R * spec.V0 ** (1 / 3) / 2 + dt * v[:, 2].clamp_max(0.0)
        J[:, 2] += spec.s_n * m / dt * (-gap).clamp_min(0.0)
        A = -dt * spec.V0 * _stress(F, Fpi, Fdot, spec, mu, lam)
        one = torch.ones((N, 1), dtype=torch.float64, device=dev)
        S = scatter((torch.cat([m * n[:, None] * one, m * n[:, None] * v, (A @ q[:, :, None])[:, :, 0] + n[:, None] * J], 1)
                     for n, q in zip(Ns, gN)), 7)
        mass = S[:, :, 0]
        inv = torch.where(mass > 0, 1 / mass.clamp_min(1e-300), torch.zeros_like(mass))[:, :, None]
        S = _couple(S[:, :, 1:], mass, codes)
        old = (S[:, :, :3] * inv).reshape(total, 3)
        new = ((S[:, :, :3] + S[:, :, 3:]) * inv).reshape(total, 3)
        so, sn = (sum(n[:, None] * u[q] for n, q in zip(Ns, rows)) for u in (old, new))
        v = spec.beta * (v - so) + sn
        x = x + dt * sn
        S = _couple(scatter((m * n[:, None] * v for n in Ns), 3), mass, codes)
        star = (S * inv).reshape(total, 3)
        G = sum(star[q][:, :, None] * gn[:, None, :] for q, gn in zip(rows, gN))
        Fdot = G
        F = F + dt * G
        fresh = ((m1 | m2) & (1 << cut)) == 0
        m1 = torch.where(fresh & (label == 1), m1 | (1 << cut), m1)
        m2 = torch.where(fresh & (label == 2), m2 | (1 << cut), m2)
        tool["x"] = tool["x"] + dt * tool["v"]
    return dict(x=x, v=v, F=F.reshape(-1, 9), mask1=m1.to(torch.int32), mask2=m2.to(torch.int32), wrench=wrench,
                forces=torch.stack(forces))


def exact(case, seed):
    """None for contact and surface: neighbour lists with pair friction and
    dual contouring are not restated here; labels are whole numbers, gradients
    would need reverse mode through all of this."""
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind in ("contact", "surface"):
        return None
    if kind == "calibration":
        st = prepare(case, seed)
        n = len(st.spec.X)
        state = dict(x=st.spec.X, v=np.zeros((n, 3)), F=np.tile(np.eye(3).ravel(), (n, 1)),
                     mask1=np.zeros(n, np.uint32), mask2=np.zeros(n, np.uint32))
        forces = _rollout64(st.spec, state, case["substeps"])["forces"]
        return {"loss": ((forces.cpu().numpy() - st.target) ** 2).sum(), "gradient": None, "forces": forces}
    if kind == "batch":
        got = [_rollout64(spec, state, case["substeps"]) for spec, state in _batch(case, rng)]
        return {"x": torch.cat([r["x"] for r in got]), "F": torch.cat([r["F"] for r in got]),
                "wrench": torch.stack([r["wrench"] for r in got])}
    r = _rollout64(*_single(case, rng), case["substeps"])
    return {k: r[k] if r[k].is_floating_point() else None for k in ("x", "v", "F", "mask1", "mask2", "wrench")}
