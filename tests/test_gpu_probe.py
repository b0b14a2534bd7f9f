"""fsi_probe_peaks as a ceiling: no product of the library is above it.  The assembled B product does 27 x 24
float64 FMAs a node (csrc/stencil.cu) and is bound by them; both rates are event-timed, 3 % apart at most for
the events and clock steps."""
import pytest

from tests.gpu_helpers import DEV, T

pytestmark = pytest.mark.gpu

import torch  # noqa: E402

from paper_2402_10348_gb300 import fsi  # noqa: E402
from tests.helpers import desc_small  # noqa: E402
from workloads import random_state  # noqa: E402


def test_the_float64_ceiling_is_above_the_b_product():
    d = desc_small(n=(64, 64, 64))
    mesh = fsi.fsi_create_mesh(d)
    fsi.fsi_set_stream(mesh)
    st = [T(a) for a in random_state(d, 0)]
    rhs = torch.randn(6 * d.nn, dtype=torch.float64, device=DEV)
    o = fsi.solve_opts(m=30, rtol=1e-30, max_iter=30)
    fsi.fsi_gmres(mesh, fsi.FSI_BLOCK_B(0), *st, rhs, torch.zeros_like(rhs), o, allow_noconv=True)
    fsi.fsi_profile(mesh, True)
    fsi.fsi_gmres(mesh, fsi.FSI_BLOCK_B(0), *st, rhs, torch.zeros_like(rhs), o, allow_noconv=True)
    launches, ms = fsi.fsi_profile_read(mesh)["b_jvp_f64"][:2]
    rate = 2.0 * 27 * 24 * d.nn * launches / (ms * 1e-3) / 1e12
    peak = fsi.fsi_probe_peaks()
    print(f"B product {rate:.3f} TFLOP/s, probe {peak}")
    assert rate <= 1.03 * peak["fp64_tflops"]
