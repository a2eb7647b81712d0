"""The cluster kernel with more samples than one round of clusters holds, with a ragged last cluster, and with the widest weight share
that it takes: the samples of the strict order (whose sums go in another order, which may move a decision that nearly ties), and the same
ones in every call."""
import pytest
import torch

import synth_inputs as si

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,H,batch", [(784, (1024, 1024), 401), (200, (500,), 1100), (1024, (1536, 1536), 260), (1936, (2048, 2048, 2048), 17)])
def test_rounds(T, H, batch):
    import __graft_entry__ as ge
    ge.build()
    import paper_2002_03629_b200 as p
    cfg = si.MadeConfig("rounds", 73, D=T, C=1, H=H, act=si.ACT_RELU, prec=si.PREC_BF16, batch=batch, noise_kind=si.NOISE_LOGISTIC, w_var_scale=1.0, b_var=0.1)
    W, b = si.made_weights(cfg)
    model = p.Model.from_config(cfg, W, b, si.made_lut(cfg))
    noise = torch.from_numpy(si.draw_noise(cfg)).cuda()
    ref = torch.empty((batch, T), dtype=torch.uint8, device="cuda")
    assert p.sequential_sample(model, noise, cfg.noise_kind, ref) == 0
    iters = torch.empty(batch, dtype=torch.int32, device="cuda")
    for mode, block in ((p.JS_JACOBI, 0), (p.JS_GS_JACOBI, T // 4)):
        first = None
        for _ in range(3):
            out = torch.full((batch, T), 7, dtype=torch.uint8, device="cuda")
            assert p.jacobi_sample(model, noise, cfg.noise_kind, None, mode, block, 0, out, iters) == 0
            assert int(iters.min()) >= 1
            first = out if first is None else first
            assert torch.equal(out, first)
        assert int((first == ref).all(1).sum()) >= batch - max(1, batch // 8)
    model.close()
