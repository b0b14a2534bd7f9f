"""fsi_batch_layout's launch count over a refined solve against the profiler's counts of the meshes.  The batch counts
what it launches itself, not each mesh's staging, diagonal and coefficients; a batched product of two
kernels (elements, node sums) is one entry of its class."""
import numpy as np
import pytest

from tests.gpu_helpers import DEV, T

pytestmark = pytest.mark.gpu

import torch  # noqa: E402

from paper_2402_10348_gb300 import fsi  # noqa: E402
from tests.helpers import desc_small  # noqa: E402
from workloads import random_state  # noqa: E402


@pytest.mark.parametrize("precision", [fsi.FSI_PREC_FP64, fsi.FSI_PREC_FP32_IR])
def test_launches_of_a_solve(precision):
    descs = [desc_small(n=n) for n in ((6, 5, 4), (9, 4, 7), (8, 8, 8))]
    meshes = [fsi.fsi_create_mesh(d) for d in descs]
    for m in meshes:
        fsi.fsi_set_stream(m)
    states = [tuple(T(a) for a in random_state(d, 1)) for d in descs]
    b = fsi.fsi_batch_create(meshes, block=fsi.FSI_BLOCK_NS, m=8)
    fsi.fsi_batch_set_graph(b, False)
    rhs = T(np.random.default_rng(3).normal(size=b.offsets[-1]))
    o = fsi.solve_opts(m=8, rtol=1e-30, max_iter=24, precision=precision, ir_max=2)
    for m in meshes:
        fsi.fsi_profile(m, True)
    before = b.layout()[2]
    fsi.fsi_batch_gmres(b, states, rhs, torch.zeros_like(rhs), o, allow_noconv=True)
    count = b.layout()[2] - before
    prof = [fsi.fsi_profile_read(m) for m in meshes]
    own = sum(v[0] for p in prof for k, v in p.items() if k not in ("stage", "op_builds", "ns_diag"))
    # the batched products run under the first mesh's class; the refinement's are each mesh's own
    products = prof[0]["ns_jvp_f64"][0] if precision == fsi.FSI_PREC_FP64 else prof[0]["ns_jvp_f32"][0]
    assert products > 0 and count == own + products
