"""One GMRES cycle at every restart-length class of the fused update (kernels are made for lengths
rounded up to 8; past 32 with other CTA sizes), single and batched, float64 and float32 basis.

A cycle's residual is the least over the Krylov space, one number whatever the basis: reference is
a modified Gram-Schmidt cycle (twice orthogonalised) in torch on the products and the diagonal of fsi_jvp and fsi_diag.
Float64 agrees to 1e-8 of it.  With a float32 operator and basis each of up to 64 vectors carries float32
rounding (6e-8 of its length, a few times in a product), which reaches the residual as at most
sqrt(64) x 10 x 6e-8 = 5e-6 of the right-hand side times the coefficients' size (of order 1 to 10 here): 5e-5."""
import numpy as np
import pytest

from tests.gpu_helpers import DEV, T

pytestmark = pytest.mark.gpu

import torch  # noqa: E402

from paper_2402_10348_gb300 import fsi  # noqa: E402
from tests.helpers import desc_small  # noqa: E402
from workloads import random_state  # noqa: E402

DESCS = [desc_small(n=(24, 23, 22)), desc_small(n=(9, 6, 11), rho_inf=0.5)]  # 55,200 and 3,360 unknowns
FLAGS = fsi.FSI_ELASTIC_AUG


def _least_residuals(mesh, st, rhs, m):
    """|r_k| / |b| for k = 1..m of right-Jacobi GMRES from 0."""
    d = torch.zeros_like(rhs)
    fsi.fsi_diag(mesh, fsi.FSI_BLOCK_NS, *st, d, FLAGS)
    V = [rhs / torch.linalg.norm(rhs)]
    H = np.zeros((m + 1, m))
    out = []
    for j in range(m):
        w = torch.zeros_like(rhs)
        fsi.fsi_jvp(mesh, fsi.FSI_BLOCK_NS, *st, (V[j] / d).contiguous(), w, FLAGS)
        for _ in range(2):
            for i, v in enumerate(V):
                h = float(v @ w)
                H[i, j] += h
                w -= h * v
        H[j + 1, j] = float(torch.linalg.norm(w))
        V.append(w / H[j + 1, j])
        e = np.zeros(j + 2)
        e[0] = 1.0
        y = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)[0]
        out.append(float(np.linalg.norm(e - H[:j + 2, :j + 1] @ y)))
    return out


def test_one_cycle_at_every_length():
    meshes = [fsi.fsi_create_mesh(d) for d in DESCS]
    for m in meshes:
        fsi.fsi_set_stream(m)
    states = [tuple(T(a) for a in random_state(d, 7, amp_v=0.3)) for d in DESCS]
    rhs = [T(np.random.default_rng(3).normal(size=4 * d.nn)) for d in DESCS]
    ref = [_least_residuals(m, s, r, 64) for m, s, r in zip(meshes, states, rhs)]
    for k in (1, 7, 8, 9, 16, 24, 31, 32, 33, 40, 41, 48, 55, 56, 57, 63, 64):
        for precision, tol in ((fsi.FSI_PREC_FP64, 0.0), (fsi.FSI_PREC_FP32_IR, 5e-5)):
            o = fsi.solve_opts(m=k, rtol=1e-30, max_iter=k, precision=precision, flags=FLAGS, ir_inner_rtol=1e-30, ir_max=1)
            got = [fsi.fsi_gmres(m, fsi.FSI_BLOCK_NS, *s, r, torch.zeros_like(r), o, allow_noconv=True)
                   for m, s, r in zip(meshes, states, rhs)]
            b = fsi.fsi_batch_create(meshes, block=fsi.FSI_BLOCK_NS, m=k)
            x = torch.zeros(b.offsets[-1], dtype=torch.float64, device=DEV)
            got += fsi.fsi_batch_gmres(b, states, torch.cat(rhs), x, o, allow_noconv=True)
            for i, g in enumerate(got):
                want = ref[i % 2][k - 1]
                assert g.iterations == k, (k, precision, i)
                assert abs(g.rel_res - want) <= 1e-8 * want + tol, (k, precision, i, g.rel_res, want)
