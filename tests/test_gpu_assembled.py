"""Assembled float64 operators (node rows of 27 neighbours, built by solves) against the oracle's
products and against the direct products of fsi_jvp.

A capped solve returns x and the relative residual that the assembled operator gives; the same
residual from the other form differs only by rounding.  Two forms of an operator agree to
TOL64 = 1e-10 of the largest entry of J x (tests/test_gpu_operators.py), so the two relative
residuals differ by at most TOL64 max|J x| sqrt(n) / |rhs|."""
import math

import numpy as np
import pytest

from tests.gpu_helpers import DEV, Gpu, T

pytestmark = pytest.mark.gpu

import torch  # noqa: E402

from oracle import ac, cgt, ns  # noqa: E402
from oracle.fields import Problem, State  # noqa: E402
from oracle.tet import TetProblem  # noqa: E402
from paper_2402_10348_gb300 import fsi  # noqa: E402
from tests.helpers import desc_small  # noqa: E402
from workloads import random_state, tet_box_mesh  # noqa: E402

TOL64 = 1e-10
GAMMA, BETA = 0.37, -0.21


def _solve(d, st, block, n, aug=True):
    """(x, rhs, relative residual) of a capped solve with a random right-hand side."""
    g = Gpu(d, *st)
    fsi.fsi_set_ac_coeffs(g.mesh, 0, GAMMA, BETA)
    rhs = T(np.random.default_rng(3).normal(size=n))
    x = torch.zeros(n, dtype=torch.float64, device=DEV)
    o = fsi.solve_opts(m=8, max_iter=16, rtol=1e-14, flags=fsi.FSI_ELASTIC_AUG if aug else 0)
    info = fsi.fsi_gmres(g.mesh, block, *g.st(), rhs, x, o, allow_noconv=True)
    return g, x, rhs, info.rel_res


def _agree(rel, rhs, y):
    r = np.linalg.norm(rhs - y) / np.linalg.norm(rhs)
    assert abs(r - rel) <= TOL64 * np.abs(y).max() * math.sqrt(y.size) / np.linalg.norm(rhs), (r, rel)


# one element; one layer; node counts below, at and above a tile of 128 nodes (3 x 6 x 7 = 126,
# 4 x 4 x 8 = 128, 129 = 43 x 3 is not a box: 5 x 2 x 13 = 130); a long thin row
@pytest.mark.parametrize("n", [(1, 1, 1), (4, 3, 1), (2, 5, 6), (3, 3, 7), (4, 1, 12), (37, 2, 3), (9, 10, 8)])
@pytest.mark.parametrize("kw", [dict(), dict(n_solid=2, rho_inf=0.5), dict(dirichlet=False)])
def test_assembled_operators_match_the_oracle(n, kw):
    d = desc_small(n=n, **kw)
    st = random_state(d, 4)
    pb, os = Problem(d), State(*st)
    for aug in (True, False):
        _, x, rhs, rel = _solve(d, st, fsi.FSI_BLOCK_NS, 4 * d.nn, aug)
        _agree(rel, rhs.cpu().numpy(), ns.ns_jvp(pb, os, x.cpu().numpy().reshape(4, -1), elastic_aug=aug).ravel())
    _, x, rhs, rel = _solve(d, st, fsi.FSI_BLOCK_AC(0), d.nn)
    _agree(rel, rhs.cpu().numpy(), ac.ac_jvp(pb, os, 0, GAMMA, BETA, x.cpu().numpy()))
    s = d.n_solid - 1
    _, x, rhs, rel = _solve(d, st, fsi.FSI_BLOCK_B(s), 6 * d.nn)
    _agree(rel, rhs.cpu().numpy(), cgt.cgt_jvp(pb, os, s, x.cpu().numpy().reshape(6, -1)).ravel())


def test_assembly_in_several_slabs_of_layers():
    """A mesh whose element matrices do not fit their scratch at once."""
    d = desc_small(n=(260, 130, 17))
    st = random_state(d, 6)
    for block, n in ((fsi.FSI_BLOCK_NS, 4 * d.nn), (fsi.FSI_BLOCK_AC(0), d.nn), (fsi.FSI_BLOCK_B(0), 6 * d.nn)):
        g, x, rhs, rel = _solve(d, st, block, n)
        y = torch.zeros_like(x)
        fsi.fsi_jvp(g.mesh, block, *g.st(), x, y)
        _agree(rel, rhs.cpu().numpy(), y.cpu().numpy())


def _tet_solve(d, coords, conn, st, aug=True):
    mesh = fsi.fsi_create_tet_mesh(d, coords, conn)
    fsi.fsi_set_stream(mesh)
    dst = [T(a) for a in st]
    rhs = T(np.random.default_rng(3).normal(size=4 * d.nn))
    x = torch.zeros_like(rhs)
    o = fsi.solve_opts(m=8, max_iter=16, rtol=1e-14, flags=fsi.FSI_ELASTIC_AUG if aug else 0)
    info = fsi.fsi_gmres(mesh, fsi.FSI_BLOCK_NS, *dst, rhs, x, o, allow_noconv=True)
    return mesh, dst, x, rhs.cpu().numpy(), info.rel_res


# nodes below, at and above slices of 32 (8; 4 x 4 x 2 = 32; 60; 420)
@pytest.mark.parametrize("n,kw", [((1, 1, 1), {}), ((3, 3, 1), dict(n_solid=2)), ((4, 3, 2), dict(rho_inf=0.5)),
                                  ((9, 5, 6), dict(n_solid=2, rho_inf=0.5))])
def test_assembled_tetrahedra_match_the_oracle(n, kw):
    d = desc_small(n=n, **kw)
    st = random_state(d, 4)
    pb, os = TetProblem(d, jitter=0.25, seed=3), State(*st)
    for aug in (True, False):
        _, _, x, rhs, rel = _tet_solve(d, pb.mesh.X, pb.mesh.conn, st, aug)
        _agree(rel, rhs, ns.ns_jvp(pb, os, x.cpu().numpy().reshape(4, -1), elastic_aug=aug).ravel())


def test_tetrahedra_with_a_row_too_long_for_the_slices():
    """Node 0 shares elements with more nodes than a row holds: the element matrices are applied."""
    d = desc_small(n=(6, 6, 6))
    X, conn = tet_box_mesh(d, 0.1, 5)
    others = np.random.default_rng(0).permutation(np.arange(1, d.nn))[: (d.nn - 1) // 3 * 3].reshape(-1, 3)
    extra = np.concatenate([np.zeros((len(others), 1), dtype=conn.dtype), others], axis=1)
    e = [X[:, extra[:, a]] - X[:, extra[:, 0]] for a in (1, 2, 3)]
    vol = np.einsum("ie,ie->e", e[0], np.cross(e[1].T, e[2].T).T)
    extra[vol < 0] = extra[vol < 0][:, [0, 2, 1, 3]]
    extra = extra[np.abs(vol) > 1e-6]
    assert 3 * len(extra) > 100
    mesh, dst, x, rhs, rel = _tet_solve(d, X, np.concatenate([conn, extra]), random_state(d, 4))
    y = torch.zeros_like(x)
    fsi.fsi_jvp(mesh, fsi.FSI_BLOCK_NS, *dst, x, y)
    _agree(rel, rhs, y.cpu().numpy())
