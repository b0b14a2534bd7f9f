"""The assembled momentum operator on tetrahedra whose element matrices (2 KB each) exceed one slab
of 2^19 elements: the product against the direct one, with the elements in mesh order and in an order in
which every slab reaches every node, and the device memory a solve leaves allocated.

Bounds: the product as in tests/test_gpu_assembled.py (two relative residuals of forms that agree to 1e-10 of
max |J x|).  Memory: 2^19 x 2 KB = 1.07 GB of matrices, rows of at most 27 neighbours x (128 + 4) bytes a
node, and m + 9 vectors of 4 doubles a node; twice the vectors for scratch of other kinds."""
import numpy as np
import pytest

from tests.gpu_helpers import DEV, T

pytestmark = pytest.mark.gpu

import torch  # noqa: E402

from paper_2402_10348_gb300 import fsi  # noqa: E402
from tests.helpers import desc_small  # noqa: E402
from workloads import random_state, tet_box_mesh  # noqa: E402

TOL64 = 1e-10
M = 8


@pytest.mark.parametrize("shuffled", [False, True])
def test_rows_summed_in_slabs_of_elements(shuffled):
    d = desc_small(n=(72, 72, 72))
    X, conn = tet_box_mesh(d, 0.1, 5)
    if shuffled:
        conn = conn[np.random.default_rng(1).permutation(len(conn))]
    assert len(conn) > 4 << 19
    mesh = fsi.fsi_create_tet_mesh(d, X, conn)
    fsi.fsi_set_stream(mesh)
    st = [T(a) for a in random_state(d, 4)]
    rhs = T(np.random.default_rng(3).normal(size=4 * d.nn))
    x, y = torch.zeros_like(rhs), torch.zeros_like(rhs)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    info = fsi.fsi_gmres(mesh, fsi.FSI_BLOCK_NS, *st, rhs, x, fsi.solve_opts(m=M, max_iter=16, rtol=1e-14),
                         allow_noconv=True)
    torch.cuda.synchronize()
    used = free - torch.cuda.mem_get_info()[0]
    assert used <= (1 << 30) + d.nn * (27 * 132 + 2 * (M + 9) * 32), used
    fsi.fsi_jvp(mesh, fsi.FSI_BLOCK_NS, *st, x, y)
    r = float(torch.linalg.norm(rhs - y) / torch.linalg.norm(rhs))
    assert abs(r - info.rel_res) <= TOL64 * float(y.abs().max()) * rhs.numel() ** 0.5 / float(torch.linalg.norm(rhs))
