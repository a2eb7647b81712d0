"""Jacobi-GS on the CUDA cores (fp32 models, and bf16 models whose positions have neither one nor 256 logits) at the edges of
its tiles: 16 samples x 64 units, products in steps of 64 inputs, rows that a round of the copying threads shares."""
import pytest
import torch

import synth_inputs as si

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,H,batch", [(1, (1,), 1), (16, (64,), 8), (33, (65, 63), 17), (70, (128, 40), 16), (64, (200,), 33)])
@pytest.mark.parametrize("C,prec", [(1, si.PREC_F32), (5, si.PREC_F32), (3, si.PREC_BF16)])
def test_equals_the_strict_order(T, H, batch, C, prec):
    import __graft_entry__ as ge
    ge.build()
    import paper_2002_03629_b200 as p
    cfg = si.MadeConfig("jgs", 66, D=T, C=C, H=H, act=si.ACT_RELU, prec=prec, batch=batch,
                        noise_kind=si.NOISE_LOGISTIC if C == 1 else si.NOISE_GUMBEL, w_var_scale=3.0, b_var=0.1)
    W, b = si.made_weights(cfg)
    model = p.Model.from_config(cfg, W, b, si.made_lut(cfg))
    noise = torch.from_numpy(si.draw_noise(cfg)).cuda()
    ref = torch.full((batch, T), 9, dtype=torch.uint8, device="cuda")
    assert p.sequential_sample(model, noise, cfg.noise_kind, ref) == 0
    for block in sorted({1, max(1, T // 3), T}):
        out = torch.full((batch, T), 9, dtype=torch.uint8, device="cuda")
        it = torch.full((batch,), -1, dtype=torch.int32, device="cuda")
        assert p.jacobi_sample(model, noise, cfg.noise_kind, None, p.JS_JACOBI_GS, block, 0, out, it) == 0
        assert model.stats().path == 1
        # (a sweep sums in another order than a tile: a decision may differ where its two scores tie to the last bits)
        assert int((out == ref).all(1).sum()) >= batch - max(1, batch // 16)
        assert int(it.min()) >= 1 and int(it.max()) <= -(-T // block)
    model.close()
