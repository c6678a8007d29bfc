"""The workloads by which the library's speed is judged: what a user of the
interface-kinematics library has it do, through its public entry points.

Cell units throughout: positions and lengths are in cells, a velocity of 1 moves
a marker by cfl cells per step.  Interfaces are ellipsoids and spheres, flows
are divergence-free MAC fields (Fourier modes, a converging cellular mode) or a
uniform translation.  Step cases run an oscillating flow, cos(pi (n + 1/2) / 16)
in step n, so that the interface stays near its start however many steps are
taken; uniform flows translate it around the periodic box.
"""
import math

import numpy as np
import torch

from paper_2509_26361_gb300 import ebit, learned, slab
from paper_2509_26361_gb300 import workloads as W

PERIOD = 16   # steps of half an oscillation of a step case's flow
CFL = 0.5
FLUID = dict(sigma=0.072, rho1=998.0, rho2=1.2, mu1=1.0e-3, mu2=1.8e-5)
MODES = {"hf": ebit.EBIT_CURV_HF, "learned": ebit.EBIT_CURV_MLP_HF}


def listed():
    return [
        # One time step of a flow solver's interface: three split sweeps, the
        # volume fractions and the curvature.
        # The paper's translation test at its smallest grid; launches and latency count.
        dict(name="step_32_translation", kind="step", nx=32, ny=32, nz=32, flow="uniform", shapes=1, rmin=4.8,
             rmax=4.8, mode="hf", overlap=False),
        # A ragged box, learned curvature with height functions as fallback, in order.
        dict(name="step_97x75x61_learned", kind="step", nx=97, ny=75, nz=61, flow="fourier", shapes=5, rmin=5.0,
             rmax=11.0, mode="learned", overlap=False),
        # The Fourier-spheres workload: 128^3, eight spheres, height functions, the
        # fractions and curvature of a step overlapping the next step's sweeps.
        dict(name="step_128_spheres", kind="step", nx=128, ny=128, nz=128, flow="fourier", shapes=8, rmin=6.4,
             rmax=15.4, mode="hf", overlap=True),
        # The benchmark's headline: converging drops at 512^3, learned curvature.
        dict(name="step_512_drops", kind="step", nx=512, ny=512, nz=512, flow="drops", shapes=2, rmin=40.0, rmax=80.0,
             mode="learned", overlap=True),
        # Curvature of a whole field of fractions (from another solver's state, or
        # an evaluation): 64 ellipsoids, height functions and the network.
        dict(name="curvature_256_hf", kind="curvature", nx=256, ny=256, nz=256, shapes=64, rmin=4.0, rmax=32.0,
             mode="hf"),
        dict(name="curvature_256_learned", kind="curvature", nx=256, ny=256, nz=256, shapes=64, rmin=4.0, rmax=32.0,
             mode="learned"),
        # Training the network (forward, backward, Adam): eight mini-batches of the
        # training command's size, then the weights read back.
        dict(name="train_16384", kind="train", batch=16384, steps=8),
        # A parameter sweep: 64 independent grids of the batched configuration's sizes,
        # four steps replayed from a graph, then every instance's fractions.
        dict(name="batch_64", kind="batch", count=64, nmin=32, nmax=128, steps=4),
        # The one-fluid terms a Navier-Stokes solver takes each step (dense fields).
        dict(name="coupling_512", kind="coupling", nx=512, ny=512, nz=512, shapes=2, rmin=40.0, rmax=80.0),
        # One step of a caller that may not allocate device memory, near its size limit.
        dict(name="noalloc_61x64x67", kind="noalloc", nx=61, ny=64, nz=67, shapes=3, rmin=6.0, rmax=12.0),
        # One step of a rank of the slab decomposition: the state goes in and comes
        # back around every sweep.
        dict(name="slab_128", kind="slab", nx=128, ny=128, nz=128, shapes=8, rmin=6.4, rmax=15.4),
        # An AMR host's refinement mask, and a checkpoint: the brick store of the state,
        # restored into another context, which computes its fractions.
        dict(name="bricks_384", kind="bricks", nx=384, ny=384, nz=384, shapes=16, rmin=12.0, rmax=40.0),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "curvature", "train", "batch", "coupling", "noalloc", "slab", "bricks"])
    if kind == "train":
        return dict(kind=kind, batch=_log_int(rng, 700, 40000), steps=rng.randint(2, 8))
    if kind == "batch":
        return dict(kind=kind, count=_log_int(rng, 3, 48), nmin=rng.randint(16, 48), nmax=rng.randint(48, 112),
                    steps=rng.randint(2, 5))
    lo, hi = {"step": (32, 320), "curvature": (64, 288), "coupling": (64, 448), "noalloc": (24, 64), "slab": (32, 144),
              "bricks": (64, 384)}[kind]
    # boxes from cubes to 2:1, most axes not a multiple of 8
    n = _log_int(rng, lo, hi)
    nx, ny, nz = (max(lo, min(hi, int(n * rng.uniform(0.7, 1.3)))) for _ in range(3))
    if kind == "noalloc":
        while nx * ny * nz > 64 ** 3:
            nx, ny, nz = nx - 1, ny - 1, nz - 1
    m = min(nx, ny, nz)
    shapes = rng.randint(1, 12)
    rmax = max(4.0, rng.uniform(0.3, 0.6) * m * shapes ** (-1.0 / 3.0) * 0.6)
    case = dict(kind=kind, nx=nx, ny=ny, nz=nz, shapes=shapes, rmin=max(3.5, 0.5 * rmax), rmax=rmax)
    if kind == "step":
        case.update(flow=rng.choice(["uniform", "fourier"]), mode=rng.choice(["hf", "learned"]),
                    overlap=rng.random() < 0.5)
    elif kind == "curvature":
        case.update(mode=rng.choice(["hf", "learned"]))
    return case


# ------------------------------------------------------------------ inputs
def _axis(n, shift, centre):
    """Minimum-image distance of the lattice points i + shift from centre."""
    d = torch.arange(n, dtype=torch.float64, device="cuda") + (shift - centre)
    return d - torch.round(d / n) * n


def _level_set(n3, ells, shift=(0.0, 0.0, 0.0)):
    """max over the ellipsoids of 1 - |R^T (x - c) / a|^2, [nz, ny, nx]."""
    phi = None
    for c, a, R in ells:
        dx, dy, dz = (_axis(n3[k], shift[k], c[k]) for k in range(3))
        v = torch.ones((n3[2], n3[1], n3[0]), dtype=torch.float64, device="cuda")
        for b in range(3):
            w = [float(R[k, b]) / a[b] for k in range(3)]
            v.sub_(((w[1] * dy[:, None] + w[2] * dz[:, None, None]) + w[0] * dx).square_())
        phi = v if phi is None else torch.maximum(phi, v, out=phi)
    return phi


def _phi(n3, ells):
    """Level set at the nodes and at the three families of face centres."""
    faces = torch.empty((3, n3[2], n3[1], n3[0]), dtype=torch.float64, device="cuda")
    for a, sh in enumerate(((0.0, 0.5, 0.5), (0.5, 0.0, 0.5), (0.5, 0.5, 0.0))):
        faces[a] = _level_set(n3, ells, sh)
    return _level_set(n3, ells), faces


def _shapes(rng, n3, count, rmin, rmax, spheres=False):
    """Ellipsoids with semi-axes U[rmin, rmax] (one radius for a sphere), random
    rotations, bounding spheres three cells apart; fewer if they do not fit."""
    out = []
    for _ in range(300 * count):
        if len(out) == count:
            break
        a = rng.uniform(rmin, rmax, 3)
        if spheres:
            a[:] = a[0]
        c = rng.uniform(0.0, 1.0, 3) * n3
        far = True
        for c2, a2, _ in out:
            d = c - c2
            d -= np.round(d / n3) * n3
            far = far and math.sqrt(float(d @ d)) > a.max() + a2.max() + 3.0
        if far:
            out.append((c, a, np.eye(3) if spheres else W.random_rotation(rng)))
    return out


def _curl(A, n3):
    """Discrete curl of a potential on the edges, as three fields on the faces."""
    def d(v, axis):
        return torch.roll(v, -1, 2 - axis) - v

    return [d(A[(a + 2) % 3], (a + 1) % 3) - d(A[(a + 1) % 3], (a + 2) % 3) for a in range(3)]


def _fourier(rng, n3, modes=12, kmax=3):
    """Divergence-free field of 12 random Fourier modes, max |u| = 1."""
    cand = np.array([k for k in np.ndindex(7, 7, 7) if 1 <= np.sum((np.array(k) - kmax) ** 2) <= kmax * kmax]) - kmax
    k = cand[rng.choice(len(cand), size=modes, replace=False)]
    amp, phase = rng.normal(size=(modes, 3)), rng.uniform(0.0, 2.0 * np.pi, modes)
    A = []
    for c in range(3):
        e = []
        for a in range(3):
            x = (np.arange(n3[a]) + (0.5 if a == c else 0.0)) / n3[a]
            e.append(torch.from_numpy(np.exp(2j * np.pi * np.outer(k[:, a], x))).cuda())
        zy = (e[2] * torch.from_numpy(amp[:, c] * np.exp(1j * phase)).cuda()[:, None])[:, :, None] * e[1][:, None, :]
        zy = zy.reshape(modes, -1)
        A.append((zy.real.T.contiguous() @ e[0].imag.contiguous() + zy.imag.T.contiguous() @ e[0].real.contiguous())
                 .reshape(n3[2], n3[1], n3[0]))
    u = _curl(A, n3)
    top = max(float(v.abs().max()) for v in u)
    return [v.div_(top) for v in u]


def _drops(rng, n3, rmin, rmax):
    """Two ellipsoids on the x axis through the middle, 8 cells apart, and the
    flow that brings them together: a converging cellular mode and a tenth of a
    Fourier field."""
    ells, mid, ext = [], n3[0] / 2.0 + rng.uniform(-0.5, 0.5), []
    for _ in range(2):
        a, R = rng.uniform(rmin, rmax, 3), W.random_rotation(rng)
        ext.append(math.sqrt(float(np.sum((a * R[0]) ** 2))))
        ells.append((a, R))
    xs = (mid - 4.0 - ext[0], mid + 4.0 + ext[1])
    ells = [(np.array([x, n3[1] / 2.0, n3[2] / 2.0]), a, R) for x, (a, R) in zip(xs, ells)]
    u = [0.1 * v for v in _fourier(rng, n3)]
    w = [4.0 * math.pi / n for n in n3]
    sx = torch.sin(w[0] * (torch.arange(n3[0], dtype=torch.float64, device="cuda") - mid))
    sy = torch.sin(w[1] * (torch.arange(n3[1], dtype=torch.float64, device="cuda") - n3[1] / 2.0))
    psi = -sy[:, None] * sx / w[1]
    u[0] += torch.roll(psi, -1, 0) - psi
    u[1] -= torch.roll(psi, -1, 1) - psi
    return ells, u


def _uniform(rng, n3):
    v = rng.uniform(0.5, 1.0, 3) * rng.choice([-1.0, 1.0], 3)
    return [torch.full((n3[2], n3[1], n3[0]), float(c), dtype=torch.float64, device="cuda") for c in v]


def _scene(case, rng):
    n3 = np.array([case["nx"], case["ny"], case["nz"]])
    flow = case.get("flow", "fourier" if case["kind"] in ("noalloc", "slab") else None)
    if flow == "drops":
        ells, u = _drops(rng, n3, case["rmin"], case["rmax"])
    else:
        ells = _shapes(rng, n3, case["shapes"], case["rmin"], case["rmax"], spheres=case["kind"] == "step")
        u = None if flow is None else _uniform(rng, n3) if flow == "uniform" else _fourier(rng, n3)
    return [int(n) for n in n3], ells, u


def _grid(n3, ells, h=None):
    g = ebit.Grid(*n3, h=h)
    phi, faces = _phi(n3, ells)
    g.init(phi, faces)
    return g


def _fields(g):
    C = torch.zeros(g.shape, dtype=torch.float64, device="cuda")
    return C, torch.zeros_like(C), torch.zeros(g.shape, dtype=torch.uint8, device="cuda")


# ----------------------------------------------------------------- prepare
def prepare(case, seed):
    rng = np.random.default_rng([int(seed), 7])
    return dict(globals()["_prepare_" + case["kind"]](case, rng), kind=case["kind"])


def _prepare_step(case, rng):
    n3, ells, u = _scene(case, rng)
    g = _grid(n3, ells)
    C, kh, st = _fields(g)
    mlp = None
    if case["mode"] == "learned":
        mlp = learned.load_network()
        g.set_mlp(mlp)
    return dict(grid=g, mlp=mlp, u=u, C=C, kh=kh, st=st, n=0, mode=MODES[case["mode"]], steady=case["flow"] == "uniform",
                flags=ebit.EBIT_ASYNC if case["overlap"] else ebit.EBIT_INCREMENTAL)


def _prepare_curvature(case, rng):
    n3, ells, _ = _scene(case, rng)
    g = _grid(n3, ells)
    C, kh, st = _fields(g)
    g.front2vof(C, ebit.EBIT_FULL)
    mlp = learned.load_network()
    g.set_mlp(mlp)
    return dict(grid=g, mlp=mlp, C=C, kh=kh, st=st, mode=MODES[case["mode"]])


def _prepare_train(case, rng):
    # labelled stencils of spheres of 3 to 16 cells: kappa h = 2 / R of the sphere
    # whose surface is nearest
    n3 = (160, 160, 160)
    ells = _shapes(rng, np.array(n3), 40, 3.0, 16.0, spheres=True)
    g = _grid(n3, ells)
    C = torch.zeros(g.shape, dtype=torch.float64, device="cuda")
    g.front2vof(C, ebit.EBIT_FULL)
    cells = torch.nonzero(((C > 0) & (C < 1)).reshape(-1)).reshape(-1)
    p = torch.stack([cells % n3[0], cells // n3[0] % n3[1], cells // (n3[0] * n3[1])], 1) + 0.5
    c = torch.from_numpy(np.array([e[0] for e in ells])).cuda()
    r = torch.from_numpy(np.array([e[1][0] for e in ells])).cuda()
    d = p[:, None, :] - c
    d = d - torch.round(d / 160.0) * 160.0
    t = (2.0 / r[(d.norm(dim=2) - r).abs().argmin(1)]).float().contiguous()
    mlp = ebit.Mlp(learned.init_params(int(rng.integers(1 << 30))))
    X = mlp.gather(C, n3, cells.to(torch.int32))
    g.close()
    idx = [torch.from_numpy(rng.integers(0, t.numel(), case["batch"]).astype(np.int32)).cuda()
           for _ in range(case["steps"])]
    loss = torch.zeros(case["steps"], dtype=torch.float32, device="cuda")
    return dict(mlp=mlp, X=X, t=t, idx=idx, loss=loss)


def _prepare_batch(case, rng):
    # the sizes belong to the case, the interfaces and flows to the seed
    pick = np.random.default_rng([case["count"], case["nmin"], case["nmax"]])
    sizes = [32, 48, 64, 96, 128] if (case["nmin"], case["nmax"]) == (32, 128) else None
    n3s, ells, u = [], [], []
    for _ in range(case["count"]):
        if sizes:
            n3 = [int(pick.choice(sizes))] * 3
        else:
            n3 = [int(pick.integers(case["nmin"], case["nmax"] + 1)) for _ in range(3)]
        m = min(n3)
        n3s.append(tuple(n3))
        ells.append(_shapes(rng, np.array(n3), int(rng.integers(1, 5)), max(3.0, 0.07 * m), max(4.0, 0.15 * m), spheres=True))
        # a translation (the interface keeps its extent over any number of steps)
        # with a weak Fourier part
        u.append([a + 0.05 * b for a, b in zip(_uniform(rng, n3), _fourier(rng, n3))])
    b = ebit.Batch(n3s)
    C = []
    for i in range(len(n3s)):
        g = b.instance(i)
        phi, faces = _phi(n3s[i], ells[i])
        g.init(phi, faces)
        C.append(torch.zeros(g.shape, dtype=torch.float64, device="cuda"))
    b.set_velocity(u, [0.4 / n3[0] for n3 in n3s])
    return dict(batch=b, C=C, n=0, steps=case["steps"])


def _prepare_coupling(case, rng):
    n3, ells, _ = _scene(case, rng)
    g = _grid(n3, ells)
    C, kh, st = _fields(g)
    g.front2vof(C, ebit.EBIT_FULL)
    g.curvature(C, kh, st, mode=ebit.EBIT_CURV_HF, flags=ebit.EBIT_FULL)
    out = (torch.empty_like(C), torch.empty_like(C), torch.empty((3,) + g.shape, dtype=torch.float64, device="cuda"))
    return dict(grid=g, C=C, kh=kh, st=st, out=out)


def _prepare_noalloc(case, rng):
    n3, ells, u = _scene(case, rng)
    g = _grid(n3, ells)
    cb, s = g.get_state()
    h = g.h
    g.close()
    return dict(n3=n3, h=h, cb=cb, s=s, u=u, out=[(torch.empty_like(cb), torch.empty_like(s)) for _ in range(3)])


def _prepare_slab(case, rng):
    n3, ells, u = _scene(case, rng)
    g = _grid(n3, ells)
    cb, s = g.get_state()
    h = g.h
    g.close()
    sl = slab.Slab(n3[2], 0, 1)
    zs = torch.arange(sl.z0 - sl.halo, sl.z1 + sl.halo, device="cuda") % n3[2]
    cut = lambda a: torch.index_select(a, a.dim() - 3, zs).contiguous()
    engine = slab.GridEngine((n3[0], n3[1], sl.nz_local), h)
    return dict(slab=sl, engine=engine, cb=cut(cb), s=cut(s), u=[cut(v) for v in u])


def _prepare_bricks(case, rng):
    n3, ells, _ = _scene(case, rng)
    g = _grid(n3, ells)
    return dict(grid=g, other=ebit.Grid(*n3), C=torch.zeros(g.shape, dtype=torch.float64, device="cuda"))


# --------------------------------------------------------------------- run
def run(state):
    return globals()["_run_" + state["kind"]](state)


def _run_step(s):
    g, n = s["grid"], s["n"]
    lam = CFL if s["steady"] else CFL * math.cos(math.pi * (n + 0.5) / PERIOD)
    g.step(n, s["u"], lam * g.h)
    g.front2vof(s["C"], s["flags"])
    g.curvature(s["C"], s["kh"], s["st"], mode=s["mode"], flags=s["flags"])
    s["n"] = n + 1
    return {"C": s["C"], "kh": s["kh"], "st": s["st"]}


def _run_curvature(s):
    s["grid"].curvature(s["C"], s["kh"], s["st"], mode=s["mode"], flags=ebit.EBIT_FULL)
    return {"kh": s["kh"], "st": s["st"]}


def _run_train(s):
    for k, idx in enumerate(s["idx"]):
        s["mlp"].train_step(s["X"], s["t"], 1e-3, s["loss"][k:k + 1], idx=idx)
    return {"loss": s["loss"], "params": s["mlp"].get_params()}


def _run_batch(s):
    b = s["batch"]
    b.run(s["n"], s["steps"])
    s["n"] += s["steps"]
    for i, C in enumerate(s["C"]):
        b.instance(i).front2vof(C)
    return s["C"]


def _run_coupling(s):
    rho, mu, f = s["grid"].one_fluid(s["C"], s["kh"], s["st"], out=s["out"], **FLUID)
    return {"rho": rho, "mu": mu, "force": f}


def _run_noalloc(s):
    cb, sv = s["cb"], s["s"]
    for d in range(3):
        cbo, so = s["out"][d]
        ebit.ebit_advect_sweep_noalloc(s["n3"], s["h"], d, cb, sv, s["u"][d], CFL * s["h"], cbo, so)
        cb, sv = cbo, so
    return {"cb": cb, "s": sv}


def _run_slab(s):
    cb, sv = slab.run_steps(s["slab"], s["engine"], s["cb"], s["s"], s["u"], [CFL])
    return {"cb": cb, "s": sv}


def _run_bricks(s):
    mask, count = s["grid"].refine_mask()
    store = s["grid"].pack_bricks()
    s["other"].unpack_bricks(store)
    s["other"].front2vof(s["C"], ebit.EBIT_FULL)
    return {"mask": mask, "count": count, "bg": store["bg"], "C": s["C"]}


# -------------------------------------------------------------------- work
def _surface(case):
    """Surface of the shapes in cells^2, from their mean radius."""
    r = 0.5 * (case["rmin"] + case["rmax"])
    return 4.0 * math.pi * r * r * case["shapes"]


def work(case):
    """Bytes and operations that the path cannot do without.  A surface of A
    cells^2 carries 1.5 A markers and crosses about 2 A cells."""
    if case["kind"] == "train":
        rows = case["batch"] * case["steps"]
        return {"bytes": 136.0 * rows + 24.0 * 24961 * case["steps"], "flops": 1.2e5 * rows}
    if case["kind"] == "batch":
        m = 0.5 * (case["nmin"] + case["nmax"])
        area = case["count"] * 2.5 * 4.0 * math.pi * (0.11 * m) ** 2
        return {"bytes": area * (case["steps"] * 3 * (1.5 * 24 + 8) + 16.0), "flops": area * case["steps"] * 3 * 180.0}
    area, N = _surface(case), float(case["nx"]) * case["ny"] * case["nz"]
    sweep = 1.5 * 24 + 2 * 4   # per cell^2: offset in and out, velocity; colours of the cells around
    if case["kind"] == "step":
        # fractions of the cut cells written, read back with their neighbours, curvature written
        return {"bytes": area * (3 * sweep + 2 * (8 + 8 + 9)),
                "flops": area * (3 * 180.0 + 2 * (300.0 + (4.0e4 if case["mode"] == "learned" else 200.0)))}
    if case["kind"] == "curvature":
        return {"bytes": 17.0 * N, "flops": 2 * area * (4.0e4 if case["mode"] == "learned" else 200.0)}
    if case["kind"] == "coupling":
        return {"bytes": 48.0 * N + 9.0 * 2 * area, "flops": 2 * area * 30.0}
    if case["kind"] == "noalloc":
        # the state (colour byte, three offsets) and the velocity read, the state written
        return {"bytes": 3 * N * (25 + 25) + 3 * area * 12.0, "flops": 3 * area * 180.0}
    if case["kind"] == "slab":
        return {"bytes": 3 * N * (25 + 25) + 3 * area * 12.0, "flops": 3 * area * 180.0}
    # bricks: the colours read, the mask and the restored state (both its buffers) written
    # and the fractions, and the band's offsets into the store and back
    return {"bytes": (2.0 + 2 * 25 + 8) * N + 8.0 * area * 3 * 25.0, "flops": 2 * area * 300.0}


# ------------------------------------------------------------------- exact
def exact(case, seed):
    """The same results in 64-bit arithmetic with plain tensor operations; None
    for the advected states and their fractions, which have no closed form."""
    f = {"curvature": _exact_curvature, "train": _exact_train, "coupling": _exact_coupling}.get(case["kind"])
    return None if f is None else f(case, int(seed))


def _network(p, x):
    W1, b1 = p[:8192].reshape(128, 64), p[8192:8320]
    W2, b2, w3, b3 = p[8320:24704].reshape(128, 128), p[24704:24832], p[24832:24960], p[24960]
    return torch.relu(torch.relu(x @ W1.T + b1) @ W2.T + b2) @ w3 + b3


def _block(C, cells, half):
    """C around each cell, offsets -half .. half along z, y, x: a gather function."""
    nz, ny, nx = C.shape
    x, y, z = cells % nx, cells // nx % ny, cells // (nx * ny)

    def at(dx, dy, dz):
        return C[(z + dz) % nz, (y + dy) % ny, (x + dx) % nx]
    return at


def _youngs(v):
    """-grad C with 1-2-1 weights of blocks v [m, z, y, x]: [m, 3] (x, y, z)."""
    w = torch.tensor([1.0, 2.0, 1.0], dtype=torch.float64, device=v.device)
    n = []
    for dim, e in ((3, "mzy,z,y->m"), (2, "mzx,z,x->m"), (1, "myx,y,x->m")):
        n.append(-torch.einsum(e, v.select(dim, 2) - v.select(dim, 0), w, w))
    return torch.stack(n, 1)


def _heights(C, cells, n):
    """Height-function kappa h of the cells (0 where no axis has valid columns)."""
    at = _block(C, cells, 4)
    order = torch.argsort(-n.abs(), dim=1, stable=True)
    kap = torch.zeros(len(cells), dtype=torch.float64, device=C.device)
    ok = torch.zeros(len(cells), 3, dtype=torch.bool, device=C.device)
    val = torch.zeros(len(cells), 3, dtype=torch.float64, device=C.device)
    for d in range(3):
        t1, t2 = (1 if d == 0 else 0), (1 if d == 2 else 2)
        below = n[:, d] > 0
        eta, good = {}, torch.ones_like(below)
        for b2 in (-1, 0, 1):
            for b1 in (-1, 0, 1):
                col = []
                for m in range(-4, 5):
                    o = [0, 0, 0]
                    o[d], o[t1], o[t2] = m, b1, b2
                    col.append(at(*o))
                H = torch.stack(col).sum(0)
                good &= torch.where(below, (col[0] == 1) & (col[8] == 0), (col[0] == 0) & (col[8] == 1))
                eta[b1, b2] = torch.where(below, H - 4.5, 4.5 - H)
        hx, hy = (eta[1, 0] - eta[-1, 0]) / 2, (eta[0, 1] - eta[0, -1]) / 2
        hxx, hyy = eta[1, 0] + eta[-1, 0] - 2 * eta[0, 0], eta[0, 1] + eta[0, -1] - 2 * eta[0, 0]
        hxy = (eta[1, 1] - eta[1, -1] - eta[-1, 1] + eta[-1, -1]) / 4
        k = ((1 + hy * hy) * hxx + (1 + hx * hx) * hyy - 2 * hx * hy * hxy) / (1 + hx * hx + hy * hy) ** 1.5
        ok[:, d], val[:, d] = good, torch.where(below, -k, k)
    done = torch.zeros_like(ok[:, 0])
    for j in range(3):
        d = order[:, j:j + 1]
        use = ok.gather(1, d)[:, 0] & ~done
        kap = torch.where(use, val.gather(1, d)[:, 0], kap)
        done |= use
    return kap


def _exact_curvature(case, seed):
    s = prepare(case, seed)
    C = s["C"]
    cells = torch.nonzero(((C > 0) & (C < 1)).reshape(-1)).reshape(-1)
    at = _block(C, cells, 1)
    v = torch.stack([at(dx, dy, dz) for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)], 1)
    n = _youngs(v.reshape(-1, 3, 3, 3))
    k = _heights(C, cells, n)
    if case["mode"] == "learned":
        # reflect the axes with n < 0, order them by increasing |n|
        o = torch.argsort(n.abs(), dim=1, stable=True)
        neg = n < 0
        j = torch.arange(27, device="cuda")
        can = torch.stack([j % 3, j // 3 % 3, j // 9], 1)                  # canonical coordinates
        src = torch.zeros(len(cells), 27, 3, dtype=torch.int64, device="cuda")
        for q in range(3):
            a = o[:, q:q + 1]
            co = torch.where(neg.gather(1, a), 2 - can[:, q], can[:, q])
            src.scatter_(2, a[:, :, None].expand(-1, 27, 1), co[:, :, None])
        x = v.gather(1, src[:, :, 0] + 3 * src[:, :, 1] + 9 * src[:, :, 2]).float()
        head = x.bfloat16().float()
        tail = (x - head).bfloat16()
        inp = torch.zeros(len(cells), 64, dtype=torch.float64, device="cuda")
        inp[:, :27], inp[:, 32:59] = head, tail
        p = torch.from_numpy(np.load(learned.PARAMS_FILE).astype(np.float64)).cuda()
        y = _network(p, inp)
        # cells with C > 0 not reached from the centre through faces: a fragment
        pos = (v > 0).reshape(-1, 3, 3, 3)
        r = torch.zeros_like(pos)
        r[:, 1, 1, 1] = True
        for _ in range(27):
            g = r.clone()
            for dim in (1, 2, 3):
                g.narrow(dim, 1, 2).logical_or_(r.narrow(dim, 0, 2))
                g.narrow(dim, 0, 2).logical_or_(r.narrow(dim, 1, 2))
            r = g & pos
        frag = (r != pos).flatten(1).any(1)
        k = torch.where((y.abs() > 1) | frag, k, y)
    kh = torch.zeros_like(C)
    kh.view(-1)[cells] = k
    return {"kh": kh, "st": None}


def _exact_train(case, seed):
    s = prepare(case, seed)
    p = s["mlp"].get_params().double()
    m, v, losses = torch.zeros_like(p), torch.zeros_like(p), []
    for k, idx in enumerate(s["idx"]):
        q = p.clone().requires_grad_(True)
        x, t = s["X"][idx.long()].double(), s["t"][idx.long()].double()
        loss = (((_network(q, x) - t) / t.abs().clamp_min(0.05)) ** 2).sum()
        g, = torch.autograd.grad(loss / len(t), q)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        p = p - 1e-3 * (m / (1 - 0.9 ** (k + 1))) / ((v / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8)
        losses.append(loss.detach())
    return {"loss": torch.stack(losses), "params": p}


def _exact_coupling(case, seed):
    s = prepare(case, seed)
    C, kh, st, h = s["C"], s["kh"], s["st"], s["grid"].h
    s["grid"].close()
    s["out"] = None
    ok = (st == 1) | (st == 2) | (st == 3) | (st == 5)
    kap = torch.where(ok, kh / h, 0.0)
    f = torch.empty((3,) + tuple(C.shape), dtype=torch.float64, device="cuda")
    for a in range(3):
        okn, kn = torch.roll(ok, 1, 2 - a), torch.roll(kap, 1, 2 - a)
        kf = (kap + kn) / (ok.double() + okn.double()).clamp_min_(1.0)
        f[a] = FLUID["sigma"] * kf * (C - torch.roll(C, 1, 2 - a)) / h
    return {"rho": C * FLUID["rho1"] + (1 - C) * FLUID["rho2"], "mu": C * FLUID["mu1"] + (1 - C) * FLUID["mu2"],
            "force": f}
