"""The in-order sweeps of binary bf16 masked MLPs at the edges of their jobs: 32, 64 and 128 sample rows a job (few jobs take
few rows), one short and one over, one to six hidden layers, widths that complete no unit, one unit or several at a position,
blocks that cut the groups of positions."""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from parity import check_samples

pytestmark = pytest.mark.gpu

#         T    H                        batch  blocks of Jacobi-GS
SHAPES = [(33, (64,), 31, (33, 7)), (72, (72, 24), 33, (24, 31)), (96, (96, 200), 65, (50,)), (130, (400, 40, 130), 8, (32, 129)),
          (200, (200,) * 4, 130, (8, 65)), (200, (128, 256), 390, (8, 25)), (64, (64,) * 5, 64, (21,)), (66, (72,) * 6, 129, (66, 1))]


@pytest.mark.parametrize("T,H,batch,blocks", SHAPES)
def test_sequential_and_jacobi_gs(T, H, batch, blocks):
    import __graft_entry__ as ge
    ge.build()
    import paper_2002_03629_b200 as p
    cfg = si.MadeConfig("sweep", 65, D=T, C=1, H=H, act=si.ACT_GELU_TANH if T == 130 else si.ACT_RELU, prec=si.PREC_BF16,
                        batch=batch, noise_kind=si.NOISE_UNIFORM_ICDF if T == 72 else si.NOISE_LOGISTIC, w_var_scale=3.0, b_var=0.1)
    W, b = si.made_weights(cfg)
    lut, noise = si.made_lut(cfg), si.draw_noise(cfg)
    orc = oracle.from_config(cfg, W, b, lut)
    model = p.Model.from_config(cfg, W, b, lut)
    d_noise = torch.from_numpy(noise).cuda()
    xstar = orc.sequential_batch(noise, cfg.noise_kind, threads=8)
    out = torch.full((batch, T), 255, dtype=torch.uint8, device="cuda")
    assert p.sequential_sample(model, d_noise, cfg.noise_kind, out) == 0
    check_samples(orc, out.cpu().numpy(), xstar, noise, cfg.noise_kind)
    for block in blocks:
        for init in (None, si.random_init(cfg, salt=2)):
            out = torch.full((batch, T), 255, dtype=torch.uint8, device="cuda")
            it = torch.full((batch,), -1, dtype=torch.int32, device="cuda")
            d_init = None if init is None else torch.from_numpy(init).cuda()
            assert p.jacobi_sample(model, d_noise, cfg.noise_kind, d_init, p.JS_JACOBI_GS, block, 0, out, it) == 0
            check_samples(orc, out.cpu().numpy(), xstar, noise, cfg.noise_kind)
            got = it.cpu().numpy()
            # block k is final after k + 1 iterations, and one more finds nothing changed
            assert got.min() >= 1 and got.max() <= (T + block - 1) // block + 1
    model.close()
