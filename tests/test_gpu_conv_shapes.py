"""Masked convolutions at the edges of the kernel's cuts: image rows that share a load with the row above and rows too long for
it, pixel stages of every size, ragged last tiles, several tiles per CTA, one layer (no hand-over between layers) and three."""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from parity import check_samples

pytestmark = pytest.mark.gpu

#         height, width, in_ch, ch, layers, batch
SHAPES = [(3, 64, 1, 128, 2, 2), (2, 128, 2, 64, 1, 2), (5, 64, 1, 64, 3, 2), (16, 8, 1, 64, 2, 150), (5, 32, 1, 128, 1, 90),
          (9, 16, 3, 128, 2, 3)]


@pytest.mark.parametrize("height,width,in_ch,ch,layers,batch", SHAPES)
def test_jacobi_and_row_blocks(height, width, in_ch, ch, layers, batch):
    import __graft_entry__ as ge
    ge.build()
    import paper_2002_03629_b200 as p
    cfg = si.ConvConfig("conv_shape", 66, height=height, width=width, in_ch=in_ch, ch=ch, layers=layers, C=256, batch=batch)
    W, b = si.conv_weights(cfg)
    lut, noise = si.conv_lut(cfg), si.draw_noise(cfg)
    orc = oracle.from_config(cfg, W, b, lut)
    model = p.Model.from_config(cfg, W, b, lut)
    d_noise = torch.from_numpy(noise).cuda()
    some = sorted({0, batch // 2, batch - 1})
    xstar = orc.sequential_batch(noise[some], cfg.noise_kind, threads=3)
    first = None
    for mode, block in ((p.JS_JACOBI, 0), (p.JS_GS_JACOBI, 2 * width * in_ch), (p.JS_JACOBI_GS, width * in_ch)):
        out = torch.full((batch, cfg.D), 255, dtype=torch.uint8, device="cuda")
        assert p.jacobi_sample(model, d_noise, cfg.noise_kind, None, mode, block, 0, out) == 0
        x = out.cpu().numpy()
        check_samples(orc, x[some], xstar, noise[some], cfg.noise_kind)
        # one arithmetic, whatever the solver: the fixed point is the same for every image
        first = x if first is None else first
        np.testing.assert_array_equal(x, first)
    model.close()
