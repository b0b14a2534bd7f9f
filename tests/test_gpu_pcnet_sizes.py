"""The weight-gradient kernel where its work units (8 x 16 voxels of one or two planes) are ragged and
where a CTA walks several of them (1,188 units on 304 CTAs), on inputs that are known exactly: with centre-tap
identities on the finest level and zeros below, every activation there is the network's input x and
every activation gradient the loss's gradient g, so dW[co][ci][t] = sum_v g[co][v] x[ci][v + t].

Bound: bfloat16 products are exact in float32; a CTA adds at most 160 sixteens of them in turn
to an accumulator and up to 40 such sums follow, each addition off by at most 2^-22 of the sum of
magnitudes: 200 x 2^-22 = 4.8e-5 of sum |g| |x|."""
import numpy as np
import pytest

import tests.test_gpu_pcnet as base

pytestmark = pytest.mark.gpu

import torch  # noqa: E402

from oracle import pcnet as pn  # noqa: E402
from paper_2402_10348_gb300 import fsi  # noqa: E402


@pytest.mark.parametrize("n", [(8, 8, 8), (16, 15, 12), (7, 33, 19), (64, 48, 64)])
def test_weight_gradient_over_work_units(n):
    d, _, pc, _, shape, _ = base._setup(n, seed=3, linear=True)
    ws, path = [], ("enc0a", "enc0b", "dec0a", "dec0b", "out")
    for (co, ci), (name, _, _) in zip(pc.fan, pn.layer_specs(16, 4)):
        w = np.zeros((co, ci, 27))
        if name in path:
            w[np.arange(co), np.arange(co), 13] = 1.0
        ws.append(w.ravel())
    fsi.fsi_pc_set_weights(pc, np.concatenate(ws))
    x = pn.bf16(np.random.default_rng(5).normal(size=(16,) + shape))
    grad = torch.zeros(pc.n_weights, dtype=torch.float32, device=base.DEV)
    fsi.fsi_pc_grad(pc, base.to_planes(x), base.to_bf16_planar(np.zeros((4,) + shape)), grad)
    got = grad.cpu().numpy().astype(np.float64)
    _, gy = pn.loss_and_grad_y(x[:4], np.zeros((4,) + shape), base._valid_mask(d, shape))
    gy = pn.bf16(gy).reshape(4, -1)
    xp = np.pad(x, ((0, 0), (1, 1), (1, 1), (1, 1)))
    ref, mag = np.zeros((4, 16, 27)), np.zeros((4, 16, 27))
    for t in range(27):
        z, y, xx = t // 9, t // 3 % 3, t % 3
        s = xp[:, z:z + shape[0], y:y + shape[1], xx:xx + shape[2]].reshape(16, -1)
        ref[:, :, t], mag[:, :, t] = gy @ s.T, np.abs(gy) @ np.abs(s).T
    off = 0
    for (co, ci), (name, _, _) in zip(pc.fan, pn.layer_specs(16, 4)):
        dw = got[off:off + co * ci * 27].reshape(co, ci, 27)
        off += co * ci * 27
        if name in path:
            assert (np.abs(dw[:4, :16] - ref) <= 4.8e-5 * mag).all(), name
            assert not dw[4:].any() and not dw[:, 16:].any(), name
