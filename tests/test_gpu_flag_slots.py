"""Change flags of consecutive passes: models with far fewer hidden units than positions, many of whose passes have no hidden layer to compute
and so no barrier but the one at their end; Jacobi and GS-Jacobi on the grid-wide kernel, samples and iteration counts against the
oracle, the same in every call."""
import pytest
import torch

import oracle
import synth_inputs as si
from parity import check_samples

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,T,H,batch", [(256, 40, (8,), 130), (256, 65, (8, 16), 5), (1, 150, (8,), 140), (1, 96, (16,), 7)])
def test_passes_without_hidden_layers(C, T, H, batch):
    import __graft_entry__ as ge
    ge.build()
    import paper_2002_03629_b200 as p
    nk = si.NOISE_GUMBEL if C == 256 else si.NOISE_LOGISTIC
    cfg = si.MadeConfig("slots", 76, D=T, C=C, H=H, act=si.ACT_RELU, prec=si.PREC_BF16, batch=batch, noise_kind=nk, w_var_scale=6.0, b_var=0.1)
    W, b = si.made_weights(cfg)
    lut, noise = si.made_lut(cfg), si.draw_noise(cfg)
    orc = oracle.from_config(cfg, W, b, lut)
    model = p.Model.from_config(cfg, W, b, lut)
    model.set_option(p.JS_OPT_TRACE, 1)                  # (keeps binary models on the grid-wide kernel)
    d_noise = torch.from_numpy(noise).cuda()
    xstar = orc.sequential_batch(noise, nk, threads=8)
    for mode, block in ((p.JS_JACOBI, 0), (p.JS_GS_JACOBI, 1), (p.JS_GS_JACOBI, 7)):
        first = None
        for _ in range(6):
            out = torch.full((batch, T), 255, dtype=torch.uint8, device="cuda")
            it = torch.full((batch,), -1, dtype=torch.int32, device="cuda")
            assert p.jacobi_sample(model, d_noise, nk, None, mode, block, 0, out, it) == 0
            assert model.stats().path == 0
            if first is None:
                first = out, it
                audit = check_samples(orc, out.cpu().numpy(), xstar, noise, nk)
                for s in sorted(set(range(0, batch, 9)) - set(audit["excused_samples"])):
                    want = orc.jacobi(noise[s], nk)[1] if mode == p.JS_JACOBI else orc.gs_jacobi(noise[s], nk, block)[1]
                    assert int(it[s]) == want
            assert torch.equal(out, first[0]) and torch.equal(it, first[1])
    model.close()
