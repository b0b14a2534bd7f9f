"""The assembled operators' entries and diagonals, row by row, against the oracle: six steps of GMRES(1),
x += a D r, r = b - A x, a = (r, A D r) / |A D r|^2, whose x is a sum of products with A and D entry by entry.
Also from four solids on, where the element kernel takes its sum over the solids another way.

Both sides are float64 sums of a few hundred terms (relative 1e-13); six steps that do not enlarge the residual
keep them within 1e-8 of a field's largest |x|, and a wrong entry is of order one."""
import numpy as np
import pytest

from tests.gpu_helpers import DEV, T

pytestmark = pytest.mark.gpu

import torch  # noqa: E402

from oracle import blocks  # noqa: E402
from oracle.diag import block_diagonal  # noqa: E402
from oracle.fields import Problem, State  # noqa: E402
from oracle.tet import TetProblem  # noqa: E402
from paper_2402_10348_gb300 import fsi  # noqa: E402
from tests.helpers import desc_small  # noqa: E402
from workloads import random_state  # noqa: E402

COEFFS = {"gamma": {0: 0.37}, "beta": {0: -0.21}}
STEPS = 6


def _check(pb, st, mesh, dst, name, block, nc, aug=True, jacobi=True):
    nn = pb.mesh.nn
    b = np.random.default_rng(3).normal(size=nc * nn)
    D = 1.0 / block_diagonal(pb, st, name, COEFFS, aug) if jacobi else np.ones(nc * nn)
    x, r = np.zeros_like(b), b.copy()
    for _ in range(STEPS):
        q = blocks.jvp(pb, st, name, D * r, COEFFS, aug)
        a = (r @ q) / (q @ q)
        x, r = x + a * D * r, r - a * q
    got = torch.zeros(nc * nn, dtype=torch.float64, device=DEV)
    o = fsi.solve_opts(m=1, rtol=1e-30, max_iter=STEPS, precond=fsi.FSI_PC_JACOBI if jacobi else fsi.FSI_PC_NONE,
                       flags=(fsi.FSI_ELASTIC_AUG if aug else 0) | fsi.FSI_NO_STALL_STOP)
    info = fsi.fsi_gmres(mesh, block, *dst, T(b), got, o, allow_noconv=True)
    torch.cuda.synchronize()
    assert info.iterations == STEPS
    got, x = got.cpu().numpy().reshape(nc, nn), x.reshape(nc, nn)
    for c in range(nc):
        assert np.abs(got[c] - x[c]).max() <= 1e-8 * np.abs(x[c]).max(), (name, c)


def _mesh(d, st, tets=None):
    mesh = fsi.fsi_create_mesh(d) if tets is None else fsi.fsi_create_tet_mesh(d, tets.mesh.X, tets.mesh.conn)
    fsi.fsi_set_stream(mesh)
    fsi.fsi_set_ac_coeffs(mesh, 0, 0.37, -0.21)
    return mesh, [T(a) for a in st]


@pytest.mark.parametrize("n,kw", [((4, 4, 8), dict()), ((5, 2, 13), dict(n_solid=2, rho_inf=0.5, dirichlet=False)),
                                  ((5, 4, 3), dict(n_solid=4)), ((6, 3, 5), dict(n_fluid=2, n_solid=5, rho_inf=0.5))])
def test_rows_on_hexahedra(n, kw):
    d = desc_small(n=n, **kw)
    st = random_state(d, 4)
    pb, os = Problem(d), State(*st)
    mesh, dst = _mesh(d, st)
    for aug in (True, False):
        _check(pb, os, mesh, dst, "ns", fsi.FSI_BLOCK_NS, 4, aug)
    _check(pb, os, mesh, dst, ("ac", 0), fsi.FSI_BLOCK_AC(0), 1)
    s = d.n_solid - 1
    _check(pb, os, mesh, dst, ("b", s), fsi.FSI_BLOCK_B(s), 6)


def test_rows_past_the_split_kernels_nodes():
    d = desc_small(n=(33, 34, 33), n_solid=4)
    assert d.nn > 152 * 256
    st = random_state(d, 4)
    mesh, dst = _mesh(d, st)
    _check(Problem(d), State(*st), mesh, dst, "ns", fsi.FSI_BLOCK_NS, 4, jacobi=False)


@pytest.mark.parametrize("n,kw", [((3, 3, 1), dict()), ((4, 3, 2), dict(n_solid=4, rho_inf=0.5))])
def test_rows_on_tetrahedra(n, kw):
    d = desc_small(n=n, **kw)
    st = random_state(d, 4)
    pb = TetProblem(d, jitter=0.25, seed=3)
    mesh, dst = _mesh(d, st, pb)
    for aug in (True, False):
        _check(pb, State(*st), mesh, dst, "ns", fsi.FSI_BLOCK_NS, 4, aug)
