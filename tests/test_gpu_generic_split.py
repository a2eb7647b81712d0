"""fp32 models beyond the small-model kernel: the products whose inputs are dealt to the warps, at the edges of their tiles (16 rows,
32 columns, 128 inputs, 32 per warp).  Network outputs against 64 bits: fp32 sums of K products in four chains stay within
K / 4 rounding steps of 2^-24, K <= 1200 (2e-5), typically sqrt(K / 4) of them; solvers against one another bit for bit."""
import pytest
import torch

import synth_inputs as si

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,H,batch", [(500, (1100,), 1), (513, (1025, 640), 17), (784, (1024, 1024), 33), (640, (1200, 900), 5), (449, (1031, 900), 16)])
def test_outputs_and_solvers(T, H, batch):
    import __graft_entry__ as ge
    ge.build()
    import paper_2002_03629_b200 as p
    import oracle
    cfg = si.MadeConfig("split", 71, D=T, C=2, H=H, act=si.ACT_RELU, prec=si.PREC_F32, batch=batch, noise_kind=si.NOISE_LOGISTIC, w_var_scale=2.0, b_var=0.05)
    W, b = si.made_real_weights(cfg)
    model = p.Model.from_config(cfg, W, b, si.made_lut(cfg))
    orc = oracle.from_config(cfg, W, b, si.made_lut(cfg))
    x = torch.randn((batch, T), generator=torch.Generator("cuda").manual_seed(T), device="cuda")
    z = torch.empty((batch, T, 2), device="cuda")
    assert p.js_forward_logits_real(model, x, z) == 0
    for s in sorted({0, batch // 2, batch - 1}):
        want = torch.from_numpy(orc.forward_logits_real(x[s].cpu().numpy())).double()
        got = z[s].cpu().double()
        assert ((got - want).abs() / want.abs().clamp_min(want.pow(2).mean().sqrt())).max().item() <= 2e-5
    noise = torch.from_numpy(si.draw_noise(cfg)).cuda()
    seq, out = torch.empty((batch, T), device="cuda"), torch.empty((batch, T), device="cuda")
    assert p.sequential_sample_real(model, noise, seq) == 0
    for mode, block in ((p.JS_JACOBI, 0), (p.JS_GS_JACOBI, T // 3)):
        assert p.jacobi_sample_real(model, noise, None, mode, block, 0, 0.0, out) == 0
        assert model.stats().path == 1
        assert torch.equal(out, seq)
    model.close()
