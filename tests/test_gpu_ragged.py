"""bf16 masked MLPs whose widths are not multiples of 8 (rows that do not start on 16 bytes): the tensor-core kernels
serve them with padding units.  Every solver, the logits, compaction (more than one row tile) against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from parity import check_samples, logits_close

pytestmark = pytest.mark.gpu

SHAPES = [("binary", 9, (13,), 3), ("binary", 129, (250, 127), 130), ("binary", 200, (99,), 70), ("binary", 255, (256, 121, 65), 9),
          ("binary", 130, (385, 130), 300), ("cat", 7, (97,), 5), ("cat", 33, (130, 61), 70)]


@pytest.mark.parametrize("kind,T,H,batch", SHAPES)
def test_every_solver(kind, T, H, batch):
    import __graft_entry__ as ge
    ge.build()
    import paper_2002_03629_b200 as p
    C = 1 if kind == "binary" else 256
    nk = si.NOISE_LOGISTIC if C == 1 else si.NOISE_GUMBEL if T % 2 and T < 30 else si.NOISE_UNIFORM_CAT
    cfg = si.MadeConfig("ragged", 63, D=T, C=C, H=H, act=si.ACT_RELU if C == 1 else si.ACT_GELU_TANH, prec=si.PREC_BF16,
                        batch=batch, noise_kind=nk, w_var_scale=3.0, b_var=0.1)
    W, b = si.made_weights(cfg)
    lut, noise = si.made_lut(cfg), si.draw_noise(cfg)
    orc = oracle.from_config(cfg, W, b, lut)
    model = p.Model.from_config(cfg, W, b, lut)
    d_noise = torch.from_numpy(noise).cuda()
    x = si.random_init(cfg, salt=5)
    z = torch.empty((batch, T, C), device="cuda")
    assert p.js_forward_logits(model, torch.from_numpy(x).cuda(), z) == 0 and model.stats().path == 0
    n = min(batch, 4)
    err, ok = logits_close(z[:n].cpu().numpy(), np.stack([orc.forward_logits(x[s]) for s in range(n)]), 2e-2)
    assert ok, err
    xstar = orc.sequential_batch(noise, nk, threads=8)
    B = max(1, T // 3)
    runs = [(p.JS_JACOBI, 0, None), (p.JS_JACOBI, 0, si.random_init(cfg, salt=1)), (p.JS_GS_JACOBI, B, None), (p.JS_GAUSS_SEIDEL, 0, None),
            (p.JS_JACOBI_GS, B, si.random_init(cfg, salt=2))]
    for mode, block, init in runs:
        out = torch.full((batch, T), 255, dtype=torch.uint8, device="cuda")
        it = torch.full((batch,), -1, dtype=torch.int32, device="cuda")
        d_init = None if init is None else torch.from_numpy(init).cuda()
        assert p.jacobi_sample(model, d_noise, nk, d_init, mode, block, 0, out, it) == 0
        if C == 1 or mode in (p.JS_JACOBI, p.JS_GS_JACOBI):
            assert model.stats().path == 0
        audit = check_samples(orc, out.cpu().numpy(), xstar, noise, nk)
        if mode == p.JS_JACOBI:
            clean = np.setdiff1d(np.arange(batch), audit["excused_samples"])
            want = np.array([orc.jacobi(noise[s], nk, None if init is None else init[s])[1] for s in clean])
            np.testing.assert_array_equal(it.cpu().numpy()[clean], want)
    model.close()
