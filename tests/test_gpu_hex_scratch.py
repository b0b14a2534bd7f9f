"""Scratch of the element-centric float64 calls on hexahedra: calls that are captured before anything ran on
their mesh, and meshes whose contributions exceed it (2^30 bytes; 48 slots of 8 bytes an element with a
solid), which go slab by slab of layers.

A window of layers of the large mesh is a mesh of its own: away from the window's first and last plane
every entry is the same sum of the same terms in the same order, so the bits agree.  gamma and beta are held
to fsi_gamma_beta_noalloc, other kernels, at 1e-11 (tests/test_gpu_operators.py)."""
import numpy as np
import pytest

from tests.gpu_helpers import DEV, Gpu, T

pytestmark = pytest.mark.gpu

import torch  # noqa: E402

from paper_2402_10348_gb300 import fsi  # noqa: E402
from tests.helpers import desc_small  # noqa: E402
from workloads import random_state  # noqa: E402

BLOCKS = [(fsi.FSI_BLOCK_NS, 4), (fsi.FSI_BLOCK_AC(0), 1), (fsi.FSI_BLOCK_B(0), 6)]


@pytest.mark.parametrize("block,nc", BLOCKS)
def test_first_call_on_a_mesh_inside_a_capture(block, nc):
    d = desc_small(n=(9, 7, 6))
    st = random_state(d, 2)
    ref = Gpu(d, *st)
    fsi.fsi_set_ac_coeffs(ref.mesh, 0, 0.37, -0.21)
    want = ref.residual(block, nc * d.nn)
    g = Gpu(d, *st)
    fsi.fsi_set_ac_coeffs(g.mesh, 0, 0.37, -0.21)
    r = torch.zeros(nc * d.nn, dtype=torch.float64, device=DEV)
    stream = torch.cuda.Stream()
    fsi.fsi_set_stream(g.mesh, stream)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        fsi.fsi_residual(g.mesh, block, *g.st(), r)
    assert float(r.abs().max()) == 0.0
    graph.replay()
    torch.cuda.synchronize()
    assert np.array_equal(r.cpu().numpy(), want)


NX, NZ, H = 220, 130, 1.0 / 256


def _desc(nz):
    return desc_small(n=(NX, NX, nz), L=(NX * H, NX * H, nz * H), eps=1.5 * H)


def test_a_mesh_in_slabs_of_layers():
    big = _desc(NZ)
    gen = torch.Generator(device=DEV).manual_seed(1)

    def field(scale):
        return scale * torch.randn((big.ncomp, NZ + 1, (NX + 1) ** 2), dtype=torch.float64, device=DEV, generator=gen)

    x = field(0.1)
    x[4] = torch.tanh(x[4] * 5.0)
    x[5] = -x[4]
    x[6:9] += 1.0
    xn, xdn = x + field(1e-3), field(0.1)
    dx = field(1.0)
    mesh = fsi.fsi_create_mesh(big)
    fsi.fsi_set_stream(mesh)
    fsi.fsi_set_ac_coeffs(mesh, 0, 0.37, -0.21)
    out = {b: [torch.zeros(nc, *x.shape[1:], dtype=torch.float64, device=DEV) for _ in range(2)] for b, nc in BLOCKS}
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    for b, nc in BLOCKS:
        fsi.fsi_residual(mesh, b, x, xn, xdn, out[b][0])
        fsi.fsi_jvp(mesh, b, x, xn, xdn, dx[:nc].contiguous(), out[b][1])
    gb = torch.zeros(2, dtype=torch.float64, device=DEV)
    got = fsi.fsi_update_ac_coeffs(mesh, 0, x, xn, xdn)
    torch.cuda.synchronize()
    # the scratch, the increments' copies and some partial sums
    assert free - torch.cuda.mem_get_info()[0] <= (1 << 30) + 12 * 8 * big.nn + (64 << 20)
    fsi.fsi_gamma_beta_noalloc(big.nx, big.ny, big.nz, big.lx, big.ly, big.lz, big.eta, x[:3].contiguous(),
                               x[4].contiguous(), gb)
    assert got[0] == pytest.approx(float(gb[0]), rel=1e-11) and got[1] == pytest.approx(float(gb[1]), rel=1e-11)
    layers = (1 << 30) // (8 * 48 * NX * NX)
    assert 2 * layers < NZ  # slabs start at layers - 1 and its double
    for a in (layers - 7, 2 * layers - 8):
        small = _desc(12)
        w = slice(a, a + 13)
        m = fsi.fsi_create_mesh(small)
        fsi.fsi_set_stream(m)
        fsi.fsi_set_ac_coeffs(m, 0, 0.37, -0.21)
        st = [f[:, w].contiguous() for f in (x, xn, xdn)]
        for b, nc in BLOCKS:
            r = torch.zeros(nc, 13, (NX + 1) ** 2, dtype=torch.float64, device=DEV)
            y = torch.zeros_like(r)
            fsi.fsi_residual(m, b, *st, r)
            fsi.fsi_jvp(m, b, *st, dx[:nc, w].contiguous(), y)
            torch.cuda.synchronize()
            for whole, part in zip(out[b], (r, y)):
                assert torch.equal(whole[:, a + 1:a + 12], part[:, 1:12]), (a, b)
