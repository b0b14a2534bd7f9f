"""Weight gradients of many voxels with one sign (centre-tap identities and zeros as in
tests/test_gpu_pcnet_sizes.py, so inputs and gradients of every layer are known): float32 sums that only grow,
where what each addition loses adds up.

Bound, relative to sum |g| |x|: an accumulator takes at most L = voxels / (16 x 912) tensor-core additions in
turn (456 for the layer of 32 channels), each of which may cut one unit of the last place, 2^-23; then at most
L_c + 42 rounded additions (groups of a CTA, blocks, warps), 2^-24 each, L_c = 8."""
import numpy as np
import pytest

import tests.test_gpu_pcnet as base

pytestmark = pytest.mark.gpu

import torch  # noqa: E402

from oracle import pcnet as pn  # noqa: E402
from paper_2402_10348_gb300 import fsi  # noqa: E402


def test_sums_of_one_sign():
    d, _, pc, _, shape, _ = base._setup((128, 128, 96), seed=3, linear=True)
    ws, path = [], ("enc0a", "enc0b", "dec0a", "dec0b", "out")
    for (co, ci), (name, _, _) in zip(pc.fan, pn.layer_specs(16, 4)):
        w = np.zeros((co, ci, 27))
        if name in path:
            w[np.arange(co), np.arange(co), 13] = 1.0
        ws.append(w.ravel())
    fsi.fsi_pc_set_weights(pc, np.concatenate(ws))
    x = pn.bf16(np.abs(np.random.default_rng(5).normal(size=(16,) + shape)))
    grad = torch.zeros(pc.n_weights, dtype=torch.float32, device=base.DEV)
    fsi.fsi_pc_grad(pc, base.to_planes(x), base.to_bf16_planar(np.zeros((4,) + shape)), grad)
    got = grad.cpu().numpy().astype(np.float64)
    _, gy = pn.loss_and_grad_y(x[:4], np.zeros((4,) + shape), base._valid_mask(d, shape))
    gy = torch.tensor(pn.bf16(gy).reshape(4, -1), device=base.DEV)
    xp = torch.nn.functional.pad(torch.tensor(x, dtype=torch.float64, device=base.DEV), (1,) * 6)
    ref = torch.zeros(4, 16, 27, dtype=torch.float64, device=base.DEV)
    for t in range(27):
        z, y, xx = t // 9, t // 3 % 3, t % 3
        ref[:, :, t] = gy @ xp[:, z:z + shape[0], y:y + shape[1], xx:xx + shape[2]].reshape(16, -1).T
    ref = ref.cpu().numpy()
    assert (ref >= 0).all()  # (so it is sum |g| |x| too)
    V, off = int(np.prod(shape)), 0
    for (co, ci), (name, _, _) in zip(pc.fan, pn.layer_specs(16, 4)):
        dw = got[off:off + co * ci * 27].reshape(co, ci, 27)[:4, :16]
        off += co * ci * 27
        if name in path:
            chain = -(-V // (16 * (912 if ci == 16 else 456)))
            assert (np.abs(dw - ref) <= (chain * 2.0 ** -23 + 50 * 2.0 ** -24) * ref).all(), name
