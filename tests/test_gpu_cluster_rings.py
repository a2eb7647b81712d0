"""The weight rings of the cluster kernel: models whose rings are short (many units or samples per cluster), tiles of one, two, odd and
even numbers of K blocks, more than 32 tiles in a layer.  Weights arrive in any order (cold L2 on the first pass); every call has
to give the samples of small batches."""
import pytest
import torch

import synth_inputs as si

pytestmark = pytest.mark.gpu

#         T     H                   batch
SHAPES = [(300, (2600, 1000), 30), (784, (2560,), 40), (1296, (2048, 2048, 1800), 16), (64, (65,), 9), (200, (130, 70), 300),
          (784, (1024, 1024), 288), (2000, (1500, 1400), 24), (900, (3000, 2000), 20)]


@pytest.mark.parametrize("T,H,batch", SHAPES)
def test_every_call_gives_the_same(T, H, batch):
    import __graft_entry__ as ge
    ge.build()
    import paper_2002_03629_b200 as p
    cfg = si.MadeConfig("rings", 68, D=T, C=1, H=H, act=si.ACT_RELU, prec=si.PREC_BF16, batch=batch, noise_kind=si.NOISE_LOGISTIC, w_var_scale=1.0, b_var=0.1)
    W, b = si.made_weights(cfg)
    model = p.Model.from_config(cfg, W, b, si.made_lut(cfg))
    noise = torch.from_numpy(si.draw_noise(cfg)).cuda()
    flush = torch.empty(160 << 20, dtype=torch.uint8, device="cuda")
    for mode, block in ((p.JS_JACOBI, 0), (p.JS_GS_JACOBI, max(1, T // 4))):
        # a few samples at a time, whose rings are long: a sample's sums do not depend on who shares its cluster
        ref = torch.empty((batch, T), dtype=torch.uint8, device="cuda")
        for lo in range(0, batch, 8):
            hi = min(batch, lo + 8)
            few = torch.empty((hi - lo, T), dtype=torch.uint8, device="cuda")
            assert p.jacobi_sample(model, noise[lo:hi].clone(), cfg.noise_kind, None, mode, block, 0, few) == 0
            ref[lo:hi] = few
        for _ in range(12):
            flush.zero_()
            out = torch.full((batch, T), 7, dtype=torch.uint8, device="cuda")
            assert p.jacobi_sample(model, noise, cfg.noise_kind, None, mode, block, 0, out) == 0
            assert model.stats().path == 0
            assert torch.equal(out, ref)
    model.close()
