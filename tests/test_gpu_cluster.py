"""The cluster kernel of binary bf16 masked MLPs at the edges of its tiles: one and three hidden layers, widths around the
64 units of a tile, every cluster size, one sample, batches that leave the last cluster ragged, blocks that cut tiles."""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from parity import check_samples

pytestmark = pytest.mark.gpu

#         T    H             batch   (cluster size: 1, 2, 4 or 8 CTAs for up to 2, 4, 8, 48 tiles in the widest layer)
SHAPES = [(5, (3,), 1), (64, (64, 128), 65), (129, (191, 65), 9), (200, (256, 512, 130), 33), (250, (700,), 120), (530, (513, 1025), 100),
          (600, (520, 776, 640), 8)]


@pytest.mark.parametrize("T,H,batch", SHAPES)
@pytest.mark.parametrize("skip", [1, 0])
def test_jacobi_and_blocks(T, H, batch, skip):
    import __graft_entry__ as ge
    ge.build()
    import paper_2002_03629_b200 as p
    cfg = si.MadeConfig("cluster", 64, D=T, C=1, H=H, act=si.ACT_GELU_TANH if T == 250 else si.ACT_RELU, prec=si.PREC_BF16,
                        batch=batch, noise_kind=si.NOISE_UNIFORM_ICDF if T == 129 else si.NOISE_LOGISTIC, w_var_scale=3.0, b_var=0.1)
    W, b = si.made_weights(cfg)
    lut, noise = si.made_lut(cfg), si.draw_noise(cfg)
    orc = oracle.from_config(cfg, W, b, lut)
    model = p.Model.from_config(cfg, W, b, lut)
    model.set_option(p.JS_OPT_FRONTIER_SKIP, skip)
    d_noise = torch.from_numpy(noise).cuda()
    xstar = orc.sequential_batch(noise, cfg.noise_kind, threads=8)
    some = sorted({0, batch // 2, batch - 1})
    for mode, block, init in ((p.JS_JACOBI, 0, None), (p.JS_JACOBI, 0, si.random_init(cfg, salt=2)),
                              (p.JS_GS_JACOBI, max(1, T // 3), None), (p.JS_GS_JACOBI, min(T, 70), si.random_init(cfg, salt=3))):
        out = torch.full((batch, T), 255, dtype=torch.uint8, device="cuda")
        it = torch.full((batch,), -1, dtype=torch.int32, device="cuda")
        d_init = None if init is None else torch.from_numpy(init).cuda()
        assert p.jacobi_sample(model, d_noise, cfg.noise_kind, d_init, mode, block, 0, out, it) == 0
        assert model.stats().path == 0
        audit = check_samples(orc, out.cpu().numpy(), xstar, noise, cfg.noise_kind)
        got = it.cpu().numpy()
        for s in some:
            if s in audit["excused_samples"]:
                continue
            i0 = None if init is None else init[s]
            want = orc.jacobi(noise[s], cfg.noise_kind, i0)[1] if mode == p.JS_JACOBI else orc.gs_jacobi(noise[s], cfg.noise_kind, block, i0)[1]
            assert got[s] == want
    if T > 64:
        out = torch.empty((batch, T), dtype=torch.uint8, device="cuda")
        assert p.jacobi_sample(model, d_noise, cfg.noise_kind, None, p.JS_JACOBI, 0, 1, out) == p.JS_NOT_CONVERGED
    model.close()


@pytest.mark.parametrize("T,H,batch", [(129, (191, 65), 9), (530, (513, 1025), 100), (600, (520, 776, 640), 40)])
def test_statistics_cover_the_whole_call(T, H, batch):
    """Counters of a call whose clusters solve their samples by themselves: what the header says, and what the same call counts
    on the grid-wide kernel (which JS_OPT_TRACE selects), where the two are comparable."""
    import __graft_entry__ as ge
    ge.build()
    import paper_2002_03629_b200 as p
    cfg = si.MadeConfig("cluster", 65, D=T, C=1, H=H, act=si.ACT_RELU, prec=si.PREC_BF16, batch=batch, noise_kind=si.NOISE_LOGISTIC, w_var_scale=3.0, b_var=0.1)
    W, b = si.made_weights(cfg)
    model = p.Model.from_config(cfg, W, b, si.made_lut(cfg))
    noise = torch.from_numpy(si.draw_noise(cfg)).cuda()
    n = [T, *H, T]
    deg = [np.arange(1, T + 1), *[1 + np.arange(h) * (T - 1) // h for h in H], np.arange(1, T + 1)]
    live = [int(np.searchsorted(deg[l], deg[l + 1], side="left" if l == len(H) else "right").sum()) for l in range(len(H) + 1)]
    out = torch.empty((batch, T), dtype=torch.uint8, device="cuda")
    it = torch.empty(batch, dtype=torch.int32, device="cuda")
    for mode, block in ((p.JS_JACOBI, 0), (p.JS_GS_JACOBI, T // 3)):
        seen = []
        for trace in (0, 1):
            model.set_option(p.JS_OPT_TRACE, trace)
            assert p.jacobi_sample(model, noise, cfg.noise_kind, None, mode, block, 0, out, it) == 0
            seen.append(model.stats())
        a, grid = seen
        assert a.path == grid.path == 0
        assert a.batch_iters_max == grid.batch_iters_max == int(it.max())
        assert a.iterations <= grid.iterations and a.tiles_issued > 0
        assert (a.tiles_skipped > 0) == (mode == p.JS_GS_JACOBI)      # Jacobi passes compute every tile here
        passes = a.iterations if mode == p.JS_JACOBI else 1
        assert a.weight_bytes >= 2 * sum(live) * passes
        assert a.mma_flops >= 2 * sum(live) * int(it.sum() if mode == p.JS_JACOBI else batch)
        assert a.mma_flops <= 2 * 64 * 64 * 64 * (a.tiles_issued * max((v + 63) // 64 for v in n))
        assert a.tiles_issued >= sum((v + 63) // 64 for v in n[1:])
    model.close()
