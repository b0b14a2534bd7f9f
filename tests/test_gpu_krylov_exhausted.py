"""GMRES past the end of its Krylov space.

The momentum block of one element has 32 unknowns, so the 33rd Arnoldi vector lies in the span of the
first 32 and the second Gram-Schmidt pass leaves rounding alone: about the square of the basis type's
rounding (emulated in numpy: 1e-32 of |J z| in float64, 1e-14 in float32), never an exact zero.  A cycle of 40 steps
with a tolerance below every estimate (1e-54 and 1e-36 there) therefore runs to its end; the norm as
a difference of squares gives 0 within a few steps, which stops the cycle as a breakdown."""
import numpy as np
import pytest

from tests.gpu_helpers import DEV, T

pytestmark = pytest.mark.gpu

import torch  # noqa: E402

from paper_2402_10348_gb300 import fsi  # noqa: E402
from tests.helpers import desc_small  # noqa: E402
from workloads import random_state  # noqa: E402

M = 40
DESCS = [desc_small(n=n, dirichlet=False) for n in ((1, 1, 1), (2, 1, 1))]  # 32 and 48 unknowns


@pytest.mark.parametrize("precision", [fsi.FSI_PREC_FP64, fsi.FSI_PREC_FP32_IR])
@pytest.mark.parametrize("seed", range(4))
@pytest.mark.parametrize("batched", [False, True])
def test_an_exhausted_space_is_no_breakdown(precision, seed, batched):
    o = fsi.solve_opts(m=M, rtol=1e-60, max_iter=M, precision=precision, ir_inner_rtol=1e-60, ir_max=1)
    meshes = [fsi.fsi_create_mesh(d) for d in DESCS]
    states = [tuple(T(a) for a in random_state(d, seed)) for d in DESCS]
    rhs = [T(np.random.default_rng(3).normal(size=4 * d.nn)) for d in DESCS]
    for m in meshes:
        fsi.fsi_set_stream(m)
    if batched:
        b = fsi.fsi_batch_create(meshes, block=fsi.FSI_BLOCK_NS, m=M)
        x = torch.zeros(b.offsets[-1], dtype=torch.float64, device=DEV)
        infos = fsi.fsi_batch_gmres(b, states, torch.cat(rhs), x, o, allow_noconv=True)
    else:
        x = [torch.zeros_like(r) for r in rhs]
        infos = [fsi.fsi_gmres(m, fsi.FSI_BLOCK_NS, *s, r, v, o, allow_noconv=True)
                 for m, s, r, v in zip(meshes, states, rhs, x)]
        x = torch.cat(x)
    torch.cuda.synchronize()
    assert torch.isfinite(x).all()
    for i in infos:
        assert (i.iterations, i.restarts) == (M, 1)
