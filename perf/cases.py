"""What is timed when the speed of the library matters: calls of its public entry points as a
program that advances a fluid-structure problem makes them, from single operator calls on a
few hundred nodes to whole block solves on two million.

A case is a dict of plain values.  `kind` says what is called:
  residual  fsi_residual of one block (the right-hand side of every Newton step)
  product   fsi_jvp of one block at a new state
  solve     one Newton step of one block: residual, then fsi_gmres on its negative
            (Allen-Cahn blocks: gamma and beta first)
  step      fsi_step, a whole partitioned time step
  batch     one Newton step of the momentum block of many uneven instances (fsi_batch_gmres)
  network   the learned preconditioner's network: forward pass, and loss and weight gradient
`setting` names the physics: an enclosed lid-driven cavity with an elastic sphere, two elastic
bodies falling in an open box, or water, air, a prescribed hull and eight ice blocks.

Solves of the momentum block that run in float64 take a fixed number of iterations (restarted
GMRES reaches a tolerance at an iteration that depends on the state; an inexact Newton method
caps them); the others run to a tolerance.  States are smooth fields with diffuse interfaces
that meet the velocity conditions, as a time step leaves them, with a little nodal noise.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch
import torch.nn.functional as nnf

from paper_2402_10348_gb300 import fsi

DEV = "cuda:0"
F64 = torch.float64


def listed():
    return [
        # the smallest call: what one residual costs when launches and latency are all of it
        dict(name="residual_ns_8", kind="residual", setting="cavity", block="ns", nx=8, ny=8, nz=8, rho_inf=0.0),
        # a product at a new state on a ragged mesh, rho_inf > 0 (x^{n+alpha} is not x^{n+1})
        dict(name="product_ns_61x47x35", kind="product", setting="falling", block="ns", nx=61, ny=47, nz=35,
             rho_inf=0.5),
        # the largest mesh of the configurations, 11 indicators and 9 solids
        dict(name="product_ns_shipice", kind="product", setting="shipice", block="ns", nx=256, ny=128, nz=64,
             rho_inf=0.0),
        # the small cavity's momentum solve to a tight tolerance: many short kernels
        dict(name="solve_ns_16_f64", kind="solve", setting="cavity", block="ns", nx=16, ny=16, nz=16, rho_inf=0.0,
             ir=False, rtol=1e-12, max_iter=2000),
        # the headline mesh: most of a float64 time step is this solve
        dict(name="solve_ns_64_f64", kind="solve", setting="cavity", block="ns", nx=64, ny=64, nz=64, rho_inf=0.0,
             ir=False, rtol=0.0, max_iter=240),
        # the same block with float32 operators inside float64 refinement
        dict(name="solve_ns_64_ir", kind="solve", setting="cavity", block="ns", nx=64, ny=64, nz=64, rho_inf=0.0,
             ir=True, rtol=1e-11, max_iter=4000),
        # an indicator's block on the falling bodies' full mesh
        dict(name="solve_ac_96x96x192_f64", kind="solve", setting="falling", block="ac", nx=96, ny=96, nz=192,
             rho_inf=0.0, ir=False, rtol=1e-11, max_iter=400),
        # a solid's left Cauchy-Green tensor on the headline mesh
        dict(name="solve_b_64_f64", kind="solve", setting="cavity", block="b", nx=64, ny=64, nz=64, rho_inf=0.0,
             ir=False, rtol=1e-11, max_iter=400),
        # a whole time step with everything between the solves
        dict(name="step_32_f64", kind="step", setting="cavity", nx=32, ny=32, nz=32, rho_inf=0.0, ir=False,
             rtol=1e-10, max_iter=4000, k_max=1),
        # many small uneven problems at once
        dict(name="batch_ns_12_ir", kind="batch", count=12, pick=0, ir=True, rtol=1e-11, max_iter=4000),
        # the linear tetrahedra, six per box cell, nodes moved
        dict(name="solve_ns_tets_32_f64", kind="solve", setting="tets", block="ns", nx=32, ny=32, nz=32, rho_inf=0.0,
             ir=False, rtol=0.0, max_iter=120),
        # one forward pass and one training gradient of the preconditioner's network
        dict(name="network_64", kind="network", setting="cavity", nx=64, ny=64, nz=64, rho_inf=0.0),
    ]


def draw(rng):
    def size(lo, hi):  # spread over the logarithm
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def box(lo, hi):
        n = size(lo, hi)
        return dict(nx=n, ny=max(3, int(n * rng.uniform(0.6, 1.4))), nz=max(3, int(n * rng.uniform(0.6, 1.4))))

    kind = rng.choice(["residual", "product", "solve", "solve", "solve", "solve", "step", "batch", "tets", "network"])
    rho_inf = rng.choice([0.0, 0.0, 0.5])
    setting = rng.choice(["cavity", "falling"])
    block = rng.choice(["ns", "ac", "b"])
    if kind == "residual":
        return dict(kind=kind, setting=setting, block=block, rho_inf=rho_inf, **box(6, 90))
    if kind == "product":
        return dict(kind=kind, setting=rng.choice(["cavity", "falling", "shipice"]), block="ns", rho_inf=rho_inf,
                    **box(8, 90))
    if kind == "solve" and block == "ns":
        if rng.random() < 0.5:
            # (the falling bodies' stiffness leaves the refinement above 1e-9)
            return dict(kind=kind, setting="cavity", block="ns", rho_inf=rho_inf, ir=True, rtol=1e-11, max_iter=4000,
                        **box(10, 48))
        return dict(kind=kind, setting=setting, block="ns", rho_inf=rho_inf, ir=False, rtol=0.0,
                    max_iter=rng.randrange(40, 241), **box(10, 54))
    if kind == "solve":
        return dict(kind=kind, setting=setting, block=block, rho_inf=rho_inf, ir=rng.random() < 0.3, rtol=1e-11,
                    max_iter=400, **box(10, 80 if block == "ac" else 54))
    if kind == "step":
        return dict(kind=kind, setting=setting, rho_inf=rho_inf, ir=rng.random() < 0.5, rtol=1e-10, max_iter=4000,
                    k_max=1, **box(8, 32))
    if kind == "batch":
        return dict(kind=kind, count=rng.randrange(4, 17), pick=rng.randrange(1, 1 << 20), ir=True, rtol=1e-11,
                    max_iter=4000)
    if kind == "tets":
        return dict(kind="solve", setting="tets", block="ns", rho_inf=0.0, ir=False, rtol=0.0,
                    max_iter=rng.randrange(30, 121), **box(6, 30))
    return dict(kind=kind, setting="cavity", rho_inf=0.0, **box(12, 64))


# ------------------------------------------------------------------ problems
def _phase(rho, mu, mu_L=0.0, solid=False):
    return SimpleNamespace(rho=rho, mu=mu, mu_L=mu_L, solid=solid)


def _face(kind=1, vel=(0.0, 0.0, 0.0), priority=0):
    return SimpleNamespace(kind=kind, vel=vel, priority=priority)


def _describe(c):
    """The problem description that fsi_create_mesh takes."""
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    d = SimpleNamespace(nx=nx, ny=ny, nz=nz, gravity=(0.0, 0.0, 0.0), eta=0.2, dt=0.01, rho_inf=c["rho_inf"],
                        c_i=36.0, prescribed_box=None, pin_node=-1, fluids=1)
    h = 1.0 / max(nx, ny, nz)
    walls = [_face() for _ in range(5)]
    if c["setting"] in ("cavity", "tets"):
        d.phases = [_phase(1.0, 0.01), _phase(1.0, 0.01, 0.1, True)]
        d.faces = walls + [_face(vel=(1.0, 0.0, 0.0), priority=1)]
        d.pin_node = 0
    elif c["setting"] == "falling":
        d.phases = [_phase(1.0, 0.01), _phase(2.0, 0.01, 1e3, True), _phase(1.5, 0.01, 50.0, True)]
        d.faces = walls + [_face(kind=0)]
        d.gravity, d.eta, d.dt = (0.0, 0.0, -9.81), 0.1, 1e-3
        h *= 2.0
    else:
        d.phases = [_phase(1000.0, 1e-3), _phase(1.0, 1.8e-5), _phase(500.0, 1e-3, 1e6, True)]
        d.phases += [_phase(900.0, 1e-3, 1e6, True) for _ in range(8)]
        d.faces = walls + [_face(kind=0)]
        d.gravity, d.eta, d.dt, d.fluids = (0.0, 0.0, -9.81), 1000.0, 1e-3, 2
        h *= 4.0
    d.lx, d.ly, d.lz = nx * h, ny * h, nz * h
    if c["setting"] == "shipice":
        d.prescribed_box = ((0.1 * d.lx, 0.4 * d.ly, 0.4 * d.lz), (0.3 * d.lx, 0.6 * d.ly, 0.6 * d.lz), (0.5, 0.0, 0.0))
    d.eps = 1.5 * h
    d.nn = (nx + 1) * (ny + 1) * (nz + 1)
    d.solids = [i for i, p in enumerate(d.phases) if p.solid]
    d.ncomp = 4 + len(d.phases) + 6 * len(d.solids)
    return d


def _coords(d):
    ax = [torch.arange(n + 1, dtype=F64, device=DEV) * (length / n)
          for n, length in ((d.nx, d.lx), (d.ny, d.ly), (d.nz, d.lz))]
    z, y, x = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
    return torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)])


def _velocity_conditions(d):
    """(mask [nn], values [3][nn]) of the nodes with a prescribed velocity."""
    n = torch.arange(d.nn, device=DEV)
    i, j, k = n % (d.nx + 1), n // (d.nx + 1) % (d.ny + 1), n // ((d.nx + 1) * (d.ny + 1))
    on = [i == 0, i == d.nx, j == 0, j == d.ny, k == 0, k == d.nz]
    mask = torch.zeros(d.nn, dtype=torch.bool, device=DEV)
    vals = torch.zeros(3, d.nn, dtype=F64, device=DEV)
    for f in sorted((f for f in range(6) if d.faces[f].kind == 1), key=lambda f: (d.faces[f].priority, -f)):
        mask |= on[f]
        for a in range(3):
            vals[a][on[f]] = d.faces[f].vel[a]
    if d.prescribed_box is not None:
        lo, hi, vel = d.prescribed_box
        xyz = (i * (d.lx / d.nx), j * (d.ly / d.ny), k * (d.lz / d.nz))
        inside = torch.ones_like(mask)
        for a in range(3):
            inside &= (xyz[a] >= lo[a]) & (xyz[a] <= hi[a])
        mask |= inside
        for a in range(3):
            vals[a][inside] = vel[a]
    return mask, vals


def _state(d, seed):
    """x^{n+1}, x^n and dx/dt^n, each [ncomp][nn]."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    X = _coords(d)
    L = torch.tensor([d.lx, d.ly, d.lz], dtype=F64, device=DEV)
    s = X / L[:, None]

    def uni(n, lo, hi):
        return lo + (hi - lo) * torch.rand(n, generator=g, dtype=F64, device=DEV)

    def smooth(noise=0.01):
        out = noise * torch.randn(d.nn, generator=g, dtype=F64, device=DEV)
        for _ in range(2):
            kv, ph = uni(3, 1.0, 3.0).floor(), uni(3, 0.0, 2.0 * math.pi)
            w = torch.sin(math.pi * kv[:, None] * s + ph[:, None])
            out += torch.randn(1, generator=g, dtype=F64, device=DEV) * w[0] * w[1] * w[2]
        return out

    bubble = (4.0 * s * (1.0 - s)).prod(0)
    mask, vals = _velocity_conditions(d)
    x, rate = (torch.empty(d.ncomp, d.nn, dtype=F64, device=DEV) for _ in range(2))
    for a in range(3):
        x[a] = 0.5 * bubble * smooth() + d.faces[5].vel[a] * s[2] ** 8
        x[a][mask] = vals[a][mask]
        rate[a] = 0.5 * bubble * smooth()
        rate[a][mask] = 0.0
    x[3], rate[3] = smooth(), 0.1 * smooth()
    left = torch.ones(d.nn, dtype=F64, device=DEV)
    rad = (0.15, 0.3) if len(d.solids) < 3 else (0.08, 0.15)
    for i in d.solids:
        centre, r = uni(3, 0.25, 0.75) * L, uni(1, *rad) * L.min()
        a = 0.5 * (1.0 + torch.tanh((r - (X - centre[:, None]).norm(dim=0)) / (math.sqrt(2.0) * d.eps))) * left
        x[4 + i] = 2.0 * a - 1.0
        left = left - a
    if d.fluids == 2:
        below = 0.5 * (1.0 + torch.tanh((0.5 * d.lz - X[2]) / (math.sqrt(2.0) * d.eps)))
        x[4], x[5] = 2.0 * left * below - 1.0, 2.0 * left * (1.0 - below) - 1.0
    else:
        x[4] = 2.0 * left - 1.0
    for i in range(len(d.phases)):
        rate[4 + i] = (1.0 - x[4 + i] ** 2) * smooth()
    for q in range(6 * len(d.solids)):
        x[4 + len(d.phases) + q] = (1.0 if q % 6 < 3 else 0.0) + 0.05 * smooth()
        rate[4 + len(d.phases) + q] = 0.2 * smooth()
    return x, x - d.dt * rate, 0.9 * rate


def _tets(d, seed):
    """Six tetrahedra per box cell around its diagonal, interior nodes moved by up to 0.1 h."""
    X = _coords(d).cpu().numpy()
    rng = np.random.default_rng(seed)
    i, j, k = (np.round(X[a] * n / length).astype(np.int64)
               for a, n, length in ((0, d.nx, d.lx), (1, d.ny, d.ly), (2, d.nz, d.lz)))
    inner = (i > 0) & (i < d.nx) & (j > 0) & (j < d.ny) & (k > 0) & (k < d.nz)
    h = np.array([d.lx / d.nx, d.ly / d.ny, d.lz / d.nz])
    X[:, inner] += (0.1 * rng.uniform(-1.0, 1.0, size=X.shape) * h[:, None])[:, inner]
    cells = _hexes(d)
    paths = []
    for p in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):
        paths.append((0, 1 << p[0], (1 << p[0]) | (1 << p[1]), 7))
    conn = cells[:, np.array(paths)].reshape(-1, 4)
    e = [X[:, conn[:, a]] - X[:, conn[:, 0]] for a in (1, 2, 3)]
    flip = np.einsum("ie,ie->e", e[0], np.cross(e[1].T, e[2].T).T) < 0
    conn[flip] = conn[flip][:, [0, 2, 1, 3]]
    return X, conn


def _hexes(d):
    """(ne, 8) node numbers of the box cells, corner a = ax + 2 ay + 4 az."""
    ez, ey, ex = (a.ravel() for a in np.meshgrid(np.arange(d.nz), np.arange(d.ny), np.arange(d.nx), indexing="ij"))
    return np.stack([(ex + (a & 1)) + (d.nx + 1) * ((ey + (a >> 1 & 1)) + (d.ny + 1) * (ez + (a >> 2)))
                     for a in range(8)], axis=1).astype(np.int64)


def _block(name, d):
    """(block id, first component, components); the last indicator, the first solid."""
    if name == "ns":
        return fsi.FSI_BLOCK_NS, 0, 4
    if name == "ac":
        return fsi.FSI_BLOCK_AC(len(d.phases) - 1), 4 + len(d.phases) - 1, 1
    return fsi.FSI_BLOCK_B(0), 4 + len(d.phases), 6


def _mesh(c, d, seed):
    if c["setting"] == "tets":
        return fsi.fsi_create_tet_mesh(d, *_tets(d, seed))
    return fsi.fsi_create_mesh(d)


def _instances(c, seed):
    """The uneven cavities of a batch."""
    rng = np.random.default_rng([c["pick"], 1])
    sizes = [int(v) for v in rng.choice([16, 24, 32, 40, 48], size=c["count"])]
    return [_describe(dict(setting="cavity", nx=n, ny=n, nz=n, rho_inf=0.0)) for n in sizes], \
        [seed * 64 + i for i in range(c["count"])]


# Allen-Cahn residuals on their own take these frozen coefficients
GAMMA, BETA = 0.3, -0.2


def _options(c):
    return fsi.solve_opts(m=30, max_iter=c["max_iter"], rtol=c["rtol"], ir_max=40,
                          precision=fsi.FSI_PREC_FP32_IR if c["ir"] else fsi.FSI_PREC_FP64)


def _network_inputs(d, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    w = np.random.default_rng(seed)
    x = torch.randn(2, d.nz + 1, d.ny + 1, d.nx + 1, 8, generator=g, device=DEV).to(torch.bfloat16)
    t = torch.randn(4, d.nn, generator=g, device=DEV).to(torch.bfloat16)
    fan = [(16, 16)] * 8 + [(16, 32), (16, 16)] * 3 + [(4, 16)]
    weights = np.concatenate([w.normal(scale=math.sqrt(2.0 / (27 * ci)), size=co * ci * 27) for co, ci in fan])
    return x, t, fan, weights.astype(np.float32)


def prepare(case, seed):
    c = case
    if c["kind"] == "batch":
        ds, seeds = _instances(c, seed)
        stream = torch.cuda.Stream()
        meshes = [fsi.fsi_create_mesh(d) for d in ds]
        for m in meshes:
            fsi.fsi_set_stream(m, stream)
            fsi.fsi_set_pressure_pin(m, False)
        states = [_state(d, s) for d, s in zip(ds, seeds)]
        batch = fsi.fsi_batch_create(meshes, m=30)
        rhs, sol = (torch.zeros(batch.offsets[-1], dtype=F64, device=DEV) for _ in range(2))
        stream.wait_stream(torch.cuda.current_stream())
        return dict(c=c, ds=ds, meshes=meshes, states=states, batch=batch, rhs=rhs, sol=sol, stream=stream)
    d = _describe(c)
    mesh = _mesh(c, d, seed)
    fsi.fsi_set_stream(mesh)
    if c["kind"] == "network":
        x, t, _, w = _network_inputs(d, seed)
        pc = fsi.fsi_pc_create(mesh, linear=True, modulate=True)
        fsi.fsi_pc_set_weights(pc, w)
        return dict(c=c, pc=pc, x=x, t=t, y=torch.zeros(4, d.nn, device=DEV),
                    grad=torch.zeros(pc.n_weights, device=DEV))
    st = dict(c=c, d=d, mesh=mesh, state=_state(d, seed))
    if c["kind"] == "step":
        st["work"] = [t.clone() for t in st["state"]]
        return st
    st["id"], _, nc = _block(c["block"], d)
    st["r"], st["sol"] = (torch.zeros(nc, d.nn, dtype=F64, device=DEV) for _ in range(2))
    if c["kind"] == "product":
        g = torch.Generator(device=DEV)
        g.manual_seed(seed + 7)
        st["dx"] = torch.randn(nc, d.nn, generator=g, dtype=F64, device=DEV)
    if c["block"] == "ac":
        fsi.fsi_set_ac_coeffs(mesh, len(d.phases) - 1, GAMMA, BETA)
    if c["block"] == "ns" and c["kind"] == "solve" and d.pin_node >= 0:
        # an enclosed domain: the pressure level is set by a shift after the solve
        fsi.fsi_set_pressure_pin(mesh, False)
    return st


def run(state):
    st, c = state, state["c"]
    kind = c["kind"]
    if kind == "network":
        fsi.fsi_pc_forward(st["pc"], st["x"], st["y"])
        loss = fsi.fsi_pc_grad(st["pc"], st["x"], st["t"], st["grad"])
        return {"y": st["y"], "grad": st["grad"], "loss": loss}
    if kind == "batch":
        off = st["batch"].offsets
        with torch.cuda.stream(st["stream"]):
            for i, m in enumerate(st["meshes"]):
                fsi.fsi_residual(m, fsi.FSI_BLOCK_NS, *st["states"][i], st["rhs"][off[i]:off[i + 1]])
            st["rhs"].neg_()
            fsi.fsi_batch_gmres(st["batch"], st["states"], st["rhs"], st["sol"], _options(c), allow_noconv=True)
            for i, d in enumerate(st["ds"]):
                p = st["sol"][off[i]:off[i + 1]].view(4, -1)[3]
                p.sub_(p[d.pin_node].clone())
        torch.cuda.current_stream().wait_stream(st["stream"])
        return {"rhs": st["rhs"], "x": st["sol"]}
    d, mesh = st["d"], st["mesh"]
    if kind == "step":
        for a, b in zip(st["work"], st["state"]):
            a.copy_(b)
        info = fsi.fsi_step(mesh, *st["work"], k_max=c["k_max"], fixed_iters=True, solve=_options(c))
        return {"x": st["work"][0], "xdn": st["work"][2], "nonlinear": info.nl_iters}
    if kind == "product":
        fsi.fsi_jvp(mesh, st["id"], *st["state"], st["dx"], st["r"])
        return {"y": st["r"]}
    out = {}
    if kind == "solve" and c["block"] == "ac":
        out["gamma"], out["beta"] = fsi.fsi_update_ac_coeffs(mesh, len(d.phases) - 1, *st["state"])
    fsi.fsi_residual(mesh, st["id"], *st["state"], st["r"])
    out["r"] = st["r"]
    if kind == "residual":
        return out
    rhs = -st["r"]
    fsi.fsi_gmres(mesh, st["id"], *st["state"], rhs, st["sol"], _options(c), allow_noconv=True)
    if c["block"] == "ns" and d.pin_node >= 0:
        st["sol"][3].sub_(st["sol"][3, d.pin_node].clone())
    out["x"] = st["sol"]
    return out


def work(case):
    """Bytes: the state's planes that the block reads and the vectors in and out.  Flops: the
    element integrals once (where they are all of the call), and for a solve its iterations on
    an assembled operator (27 neighbours; 15 on tetrahedra) with one Gram-Schmidt sweep."""
    c = case
    if c["kind"] == "batch":
        ds, _ = _instances(c, 0)
        its = 300
        return {"bytes": sum(8.0 * d.nn * (3 * d.ncomp + 8) for d in ds),
                "flops": sum(d.nn * its * (2.0 * 27 * 16 + 4.0 * 4 * 15) for d in ds)}
    d = _describe(c)
    ns, n = len(d.solids), float(d.nn)
    if c["kind"] == "network":
        v, f = n, 0.0
        for _ in range(4):
            f += v * 27 * 16 * 2.0 * (2 * 16 + 3 * 16)
            v /= 8.0
        return {"bytes": n * (32 + 8 + 16), "flops": 4.0 * f}
    elems = float(d.nx * d.ny * d.nz)
    if c["kind"] == "step":
        return {"bytes": 8.0 * n * 5 * d.ncomp,
                "flops": n * (300 * (2.0 * 27 * 16 + 240) + len(d.phases) * 25 * (54 + 50) + ns * 25 * (1300 + 300))}
    read = {"ns": 4 + 3 + len(d.phases) + 6 * ns, "ac": 5, "b": 10}[c["block"]]
    nc = {"ns": 4, "ac": 1, "b": 6}[c["block"]]
    element = {"ns": 8.0 * (700 + 200 * ns), "ac": 8.0 * 130, "b": 8.0 * 400}[c["block"]] * elems
    if c["kind"] == "residual":
        return {"bytes": 8.0 * n * (2 * read + nc), "flops": element}
    if c["kind"] == "product":
        return {"bytes": 8.0 * n * (2 * read + 2 * nc), "flops": 1.5 * element}
    its = c["max_iter"] if c["rtol"] == 0.0 else {"ns": 300, "ac": 25, "b": 25}[c["block"]]
    row = {"ns": 16, "ac": 1, "b": 24}[c["block"]] * (15 if c["setting"] == "tets" else 27)
    return {"bytes": 8.0 * n * (2 * read + 3 * nc), "flops": element + n * its * (2.0 * row + 4.0 * nc * 15)}


# ------------------------------------------------------------------ the same in 64 bits
SYM = ((0, 3, 5), (3, 1, 4), (5, 4, 2))
PAIRS = ((0, 0), (1, 1), (2, 2), (0, 1), (1, 2), (0, 2))


class _Elements:
    """Shape functions at the quadrature points, weights and metric, for some of the elements."""

    def __init__(self, d, tets=None):
        def t(a):
            return torch.as_tensor(np.ascontiguousarray(a), device=DEV)

        self.d = d
        if tets is None:
            self.conn = t(_hexes(d))
            h = np.array([d.lx / d.nx, d.ly / d.ny, d.lz / d.nz])
            N, dN = np.ones((8, 8)), np.ones((8, 8, 3))
            for q in range(8):
                for a in range(8):
                    for ax in range(3):
                        up = (a >> ax & 1)
                        v = 0.5 * (1.0 + (1.0 if up == (q >> ax & 1) else -1.0) / math.sqrt(3.0))
                        N[q, a] *= v
                        for b in range(3):
                            dN[q, a, b] *= ((1.0 if up else -1.0) / h[ax]) if b == ax else v
            self.N, self.dN = t(N), t(dN)
            self.w = torch.full((self.conn.shape[0], 1), float(h.prod() / 8.0), dtype=F64, device=DEV)
            self.G = t(np.diag(4.0 / h ** 2))[None]
        else:
            X, conn = tets
            self.conn = t(conn)
            J = np.stack([X[:, conn[:, a]].T - X[:, conn[:, 0]].T for a in (1, 2, 3)], axis=2)
            inv = np.linalg.inv(J)
            g = np.concatenate([-inv.sum(1, keepdims=True), inv], axis=1)
            big, small = (5.0 + 3.0 * math.sqrt(5.0)) / 20.0, (5.0 - math.sqrt(5.0)) / 20.0
            self.N = t(np.full((4, 4), small) + np.diag([big - small] * 4))
            self.dN = t(g)
            self.w = t(np.linalg.det(J) / 24.0)[:, None]
            self.G = t(np.einsum("eki,ekj->eij", inv, inv))
        self.tets = tets is not None

    def part(self, lo, hi):
        p = object.__new__(_Elements)
        p.__dict__.update(self.__dict__)
        p.conn, p.w = self.conn[lo:hi], self.w[lo:hi]
        if self.tets:
            p.dN, p.G = self.dN[lo:hi], self.G[lo:hi]
        return p

    def val(self, u):
        return u[self.conn] @ self.N.T

    def grad(self, u):
        if self.tets:
            g = torch.einsum("ea,ead->ed", u[self.conn], self.dN)
            return [g[:, None, k].expand(-1, 4) for k in range(3)]
        g = torch.einsum("ea,qad->deq", u[self.conn], self.dN)
        return [g[0], g[1], g[2]]

    def add(self, out, f, g):
        """out_a += sum_q w (N_a f + grad N_a . g)"""
        c = (f * self.w) @ self.N
        for k in range(3):
            if self.tets:
                c = c + (g[k] * self.w).sum(1, keepdim=True) * self.dN[:, :, k]
            else:
                c = c + (g[k] * self.w) @ self.dN[:, :, k]
        out.index_add_(0, self.conn.reshape(-1), c.reshape(-1))

    def vGv(self, v):
        return sum(v[i] * self.G[:, i, j][:, None] * v[j] for i in range(3) for j in range(3))

    @property
    def GG(self):
        return (self.G ** 2).sum((1, 2))[:, None]

    @property
    def trG(self):
        return (self.G[:, 0, 0] + self.G[:, 1, 1] + self.G[:, 2, 2])[:, None]


class _Exact:
    """Residuals and products of the three kinds of block, in float64 tensors."""

    def __init__(self, d, state, tets=None, pinned=True):
        self.d, self.pinned = d, pinned
        x, xn, xdn = state
        r = d.rho_inf
        self.al, self.am = 1.0 / (1.0 + r), 0.5 * (3.0 - r) / (1.0 + r)
        self.vs = 0.5 + self.am - self.al
        self.cm = self.am / (self.vs * d.dt)
        self.x = x
        self.xa = xn + self.al * (x - xn)
        self.xa[3] = x[3]
        self.xd = xdn + self.am * (x - xn - d.dt * xdn) / (self.vs * d.dt)
        self.el = _Elements(d, tets)

    def _chunks(self):
        ne = self.el.conn.shape[0]
        for lo in range(0, ne, 1 << 17):
            yield self.el.part(lo, min(ne, lo + (1 << 17)))

    def coefficients(self, i):
        """gamma and beta of indicator i."""
        num, den = (torch.zeros(self.d.nn, dtype=F64, device=DEV) for _ in range(2))
        iF = isF = 0.0
        phi = self.xa[4 + i]
        for el in self._chunks():
            L = [el.grad(self.xa[k]) for k in range(3)]
            g = el.grad(phi)
            n2 = g[0] ** 2 + g[1] ** 2 + g[2] ** 2
            q = sum(g[j] * L[j][k] * g[k] for j in range(3) for k in range(3))
            q = torch.where(n2 < 1e-30, torch.zeros_like(q), q / torch.where(n2 < 1e-30, torch.ones_like(n2), n2))
            zero = [torch.zeros_like(q)] * 3
            el.add(num, q, zero)
            el.add(den, torch.ones_like(q), zero)
            p = el.val(phi)
            iF = iF + ((p ** 3 - p) * el.w).sum()
            isF = isF + (0.5 * (p ** 2 - 1.0).abs() * el.w).sum()
        v = (num / den).abs()[phi.abs() <= 0.9]
        gamma = float((v ** 2).mean().sqrt()) / self.d.eta if v.numel() else 0.0
        return gamma, float(iF / isF) if float(isF) != 0.0 else 0.0

    def ns(self, dx=None):
        """The residual, or with dx the Jacobian-vector product."""
        d, xa, xd = self.d, self.xa, self.xd
        out = torch.zeros(4, d.nn, dtype=F64, device=DEV)
        for el in self._chunks():
            v = [el.val(xa[k]) for k in range(3)]
            L = [el.grad(xa[k]) for k in range(3)]
            alpha = [(1.0 + el.val(xa[4 + i])) / 2.0 for i in range(len(d.phases))]
            rho = sum(a * p.rho for a, p in zip(alpha, d.phases))
            mu = sum(a * p.mu for a, p in zip(alpha, d.phases))
            gp = el.grad(xa[3])
            acc = [el.val(xd[k]) + sum(v[j] * L[k][j] for j in range(3)) for k in range(3)]
            R = [rho * acc[k] + gp[k] - rho * d.gravity[k] for k in range(3)]
            tm = (4.0 / d.dt ** 2 + el.vGv(v) + d.c_i * (mu / rho) ** 2 * el.GG) ** -0.5
            tc = 1.0 / (el.trG * tm)
            E = [0.0] * 6
            if dx is None:
                for s, i in enumerate(d.solids):
                    a = alpha[i] * d.phases[i].mu_L
                    for q in range(6):
                        E[q] = E[q] + a * (el.val(xa[4 + len(d.phases) + 6 * s + q]) - (1.0 if q < 3 else 0.0))
                f, dL, p = [rho * (acc[k] - d.gravity[k]) for k in range(3)], L, el.val(xa[3])
                adv = [[v[j] * R[k] for j in range(3)] for k in range(3)]
                cont = R
            else:
                dv = [self.al * el.val(dx[k]) for k in range(3)]
                dL = [[self.al * g for g in el.grad(dx[k])] for k in range(3)]
                p, gdp = el.val(dx[3]), el.grad(dx[3])
                f = [rho * (self.cm / self.al * dv[k] + sum(dv[j] * L[k][j] + v[j] * dL[k][j] for j in range(3)))
                     for k in range(3)]
                cont = [f[k] + gdp[k] for k in range(3)]
                adv = [[dv[j] * R[k] + v[j] * cont[k] for j in range(3)] for k in range(3)]
                cel = self.al * self.vs * d.dt / self.am
                for s, i in enumerate(d.solids):
                    a = alpha[i] * d.phases[i].mu_L * cel
                    o = 4 + len(d.phases) + 6 * s
                    B = [el.val(xa[o + q]) for q in range(6)]
                    for q, (k, l) in enumerate(PAIRS):
                        gB = el.grad(xa[o + q])
                        t = sum(dL[k][m] * B[SYM[m][l]] + B[SYM[k][m]] * dL[l][m] - dv[m] * gB[m] for m in range(3))
                        E[q] = E[q] + a * t
            div = dL[0][0] + dL[1][1] + dL[2][2]
            for k in range(3):
                g = [mu * (dL[k][j] + dL[j][k]) + E[SYM[k][j]] + tm * adv[k][j] + ((tc * rho * div - p) if j == k else 0.0)
                     for j in range(3)]
                el.add(out[k], f[k], g)
            el.add(out[3], div, [tm / rho * cont[j] for j in range(3)])
        mask, vals = _velocity_conditions(d)
        for k in range(3):
            out[k][mask] = (self.x[k] - vals[k])[mask] if dx is None else dx[k][mask]
        if self.pinned and d.pin_node >= 0:
            out[3][d.pin_node] = (self.x if dx is None else dx)[3][d.pin_node]
        return out

    def ac(self, i, gamma, beta, dx=None):
        d, xa = self.d, self.xa
        out = torch.zeros(1, d.nn, dtype=F64, device=DEV)
        kh = gamma * d.eps ** 2
        for el in self._chunks():
            v = [el.val(xa[k]) for k in range(3)]
            phi = el.val(xa[4 + i])
            tau = (4.0 / d.dt ** 2 + el.vGv(v) + 9.0 * kh ** 2 * el.GG + (gamma * (3.0 * phi ** 2 - 1.0)) ** 2) ** -0.5
            if dx is None:
                g = el.grad(xa[4 + i])
                R = el.val(self.xd[4 + i]) + sum(v[j] * g[j] for j in range(3))
                R = R + gamma * (phi ** 3 - phi - beta * 0.5 * (phi ** 2 - 1.0).abs())
            else:
                u, g = self.al * el.val(dx[0]), [self.al * t for t in el.grad(dx[0])]
                R = self.cm / self.al * u + sum(v[j] * g[j] for j in range(3))
                R = R + gamma * (3.0 * phi ** 2 - 1.0 - beta * phi * torch.sign(phi ** 2 - 1.0)) * u
            el.add(out[0], R, [kh * g[j] + tau * v[j] * R for j in range(3)])
        return out

    def b(self, s, dx=None):
        d, xa = self.d, self.xa
        out = torch.zeros(6, d.nn, dtype=F64, device=DEV)
        o = 4 + len(d.phases) + 6 * s
        for el in self._chunks():
            v = [el.val(xa[k]) for k in range(3)]
            L = [el.grad(xa[k]) for k in range(3)]
            a = (1.0 + el.val(xa[4 + d.solids[s]])) / 2.0
            tau = (4.0 / d.dt ** 2 + el.vGv(v)) ** -0.5
            src = xa[o:o + 6] if dx is None else self.al * dx
            B = [el.val(src[q]) for q in range(6)]
            for q, (k, l) in enumerate(PAIRS):
                g = el.grad(src[q])
                rate = el.val(self.xd[o + q]) if dx is None else self.cm / self.al * B[q]
                st = sum(L[k][m] * B[SYM[m][l]] + B[SYM[k][m]] * L[l][m] for m in range(3))
                R = a * (rate + sum(v[j] * g[j] for j in range(3)) - st)
                R = R + (1.0 - a) * (B[q] - (1.0 if dx is None and q < 3 else 0.0))
                el.add(out[q], R, [tau * v[j] * R for j in range(3)])
        return out


def _gmres64(A, b, inv, tol=1e-14, most=400):
    """Full GMRES with a diagonal right preconditioner (two Gram-Schmidt passes)."""
    shape, b = b.shape, b.reshape(-1)
    beta = b.norm()
    V = [b / beta]
    H = np.zeros((most + 1, most))
    for j in range(most):
        w = A((inv * V[j]).reshape(shape)).reshape(-1)
        for _ in range(2):
            for i, u in enumerate(V):
                h = torch.dot(u, w)
                w = w - h * u
                H[i, j] += float(h)
        H[j + 1, j] = float(w.norm())
        V.append(w / w.norm())
        e = np.zeros(j + 2)
        e[0] = float(beta)
        y = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)[0]
        if np.linalg.norm(e - H[:j + 2, :j + 1] @ y) <= tol * e[0]:
            break
    return (inv * sum(float(t) * u for t, u in zip(y, V))).reshape(shape)


def _diagonal(A, d, nc, at_once=False):
    """One product per residue of the node indices modulo 3 and component (at_once: the sum of a
    node's row over its own components instead, a scaling that is near the diagonal)."""
    n = torch.arange(d.nn, device=DEV)
    i, j, k = n % (d.nx + 1), n // (d.nx + 1) % (d.ny + 1), n // ((d.nx + 1) * (d.ny + 1))
    out = torch.zeros(nc, d.nn, dtype=F64, device=DEV)
    for col in range(27):
        on = (i % 3 == col % 3) & (j % 3 == col // 3 % 3) & (k % 3 == col // 9)
        for q in [slice(0, nc)] if at_once else range(nc):
            e = torch.zeros(nc, d.nn, dtype=F64, device=DEV)
            e[q, on] = 1.0
            out[q, on] = A(e)[q, on]
    return out


def _levels(x, w, fan):
    """The network (without activation functions) in float64; x: [1][16][nz][ny][nx]."""
    ws, off = [], 0
    for co, ci in fan:
        ws.append(w[off:off + co * ci * 27].view(co, ci, 3, 3, 3))
        off += co * ci * 27

    def conv(a, k):
        return nnf.conv3d(a, ws[k], padding=1)

    def interp(nf, ncs):
        P = torch.zeros(nf, ncs, dtype=F64, device=DEV)
        for i in range(nf):
            for q in ((i // 2,) if i % 2 == 0 else (i // 2, i // 2 + 1)):
                P[i, q] = 1.0 if i % 2 == 0 else 0.5
        return P

    e, ps = [], []
    for lv in range(3):
        e.append(conv(conv(x, 2 * lv), 2 * lv + 1))
        ps.append([interp(n, n // 2 + 1) for n in x.shape[2:]])
        x = torch.einsum("bkzyx,zc,yd,xe->bkcde", e[lv], *ps[lv]) / 8.0
    x = conv(conv(x, 6), 7)
    for k, lv in ((8, 2), (10, 1), (12, 0)):
        up = torch.einsum("bkcde,zc,yd,xe->bkzyx", x, *ps[lv])
        x = conv(conv(torch.cat([e[lv], up], dim=1), k), k + 1)
    return conv(x, 14)


def exact(case, seed):
    c = case
    if c["kind"] == "step":
        return None
    if c["kind"] == "batch":
        ds, seeds = _instances(c, seed)
        r = [_Exact(d, _state(d, s), pinned=False).ns().reshape(-1) for d, s in zip(ds, seeds)]
        return {"rhs": -torch.cat(r), "x": None}
    d = _describe(c)
    if c["kind"] == "network":
        x, t, fan, w = _network_inputs(d, seed)
        w = torch.tensor(w, dtype=F64, device=DEV, requires_grad=True)
        y = _levels(x.double().permute(0, 4, 1, 2, 3).reshape(1, 16, *x.shape[1:4]), w, fan).reshape(4, -1)
        mask, _ = _velocity_conditions(d)
        rows = (~mask).double()[None].repeat(4, 1)
        rows[3] = 1.0
        rows[3, d.pin_node] = 0.0
        loss = (((y - t.double()) ** 2) * rows).sum() / rows.sum()
        loss.backward()
        return {"y": y.detach(), "grad": w.grad, "loss": float(loss.detach())}
    tets = _tets(d, seed) if c["setting"] == "tets" else None
    ex = _Exact(d, _state(d, seed), tets, pinned=c["kind"] != "solve")
    last = len(d.phases) - 1
    if c["kind"] == "product":
        g = torch.Generator(device=DEV)
        g.manual_seed(seed + 7)
        return {"y": ex.ns(torch.randn(4, d.nn, generator=g, dtype=F64, device=DEV))}
    out, gb = {}, (GAMMA, BETA)
    if c["kind"] == "solve" and c["block"] == "ac":
        gb = out["gamma"], out["beta"] = ex.coefficients(last)
    apply = {"ns": ex.ns, "ac": lambda dx=None: ex.ac(last, *gb, dx), "b": lambda dx=None: ex.b(0, dx)}[c["block"]]
    out["r"] = apply()
    if c["kind"] == "residual":
        return out
    if c["block"] != "ns":
        scale = _diagonal(apply, d, 6, at_once=True) if c["block"] == "b" else torch.ones_like(out["r"])
        out["x"] = _gmres64(apply, -out["r"], 1.0 / scale.reshape(-1))
    elif c["rtol"] > 0.0 and d.nn <= 6000:
        out["x"] = _gmres64(apply, -out["r"], 1.0 / _diagonal(apply, d, 4).reshape(-1))
        if d.pin_node >= 0:
            out["x"][3] -= out["x"][3, d.pin_node].clone()
    else:
        out["x"] = None
    return out
