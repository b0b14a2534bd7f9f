"""A float64 solve takes its products one way: direct ones if it may take few, else the assembled operator from
the first product on (its diagonal comes with it).  A solve takes a product an iteration and one a cycle for the
true residual; one that starts direct and assembles for its last product pays for both."""
import pytest

from tests.gpu_helpers import DEV, T

pytestmark = pytest.mark.gpu

import torch  # noqa: E402

from paper_2402_10348_gb300 import fsi  # noqa: E402
from tests.helpers import desc_small  # noqa: E402
from workloads import random_state, tet_box_mesh  # noqa: E402

BLOCKS = [(fsi.FSI_BLOCK_NS, 4), (fsi.FSI_BLOCK_AC(0), 1), (fsi.FSI_BLOCK_B(0), 6)]


@pytest.mark.parametrize("tets", [False, True])
@pytest.mark.parametrize("m", [1, 3, 30])
def test_direct_or_assembled(m, tets):
    d = desc_small(n=(6, 5, 4))
    mesh = fsi.fsi_create_tet_mesh(d, *tet_box_mesh(d, 0.1, 5)) if tets else fsi.fsi_create_mesh(d)
    fsi.fsi_set_stream(mesh)
    fsi.fsi_set_ac_coeffs(mesh, 0, 0.37, -0.21)
    st = [T(a) for a in random_state(d, 0)]
    for block, nc in BLOCKS[:1] if tets else BLOCKS:
        rhs = torch.randn(nc * d.nn, dtype=torch.float64, device=DEV)
        for its in range(1, 9):
            o = fsi.solve_opts(m=m, rtol=1e-30, max_iter=its, flags=fsi.FSI_ELASTIC_AUG | fsi.FSI_NO_STALL_STOP)
            fsi.fsi_profile(mesh, True)
            fsi.fsi_gmres(mesh, block, *st, rhs, torch.zeros_like(rhs), o, allow_noconv=True)
            p = fsi.fsi_profile_read(mesh)
            fsi.fsi_profile(mesh, False)
            # (direct products: the momentum block's class, elsewhere the sums of their contributions)
            direct = p["ns_jvp_f64"][0] if nc == 4 else p["node_sums"][0]
            built = p["op_builds"][0]
            assert (direct == 0) != (built == 0), (block, m, its, direct, built)
