"""Binary bf16 masked MLPs on the GRID-WIDE tensor-core kernel, which the cluster kernel leaves only deeper, wider or larger calls:
four hidden layers, or the same shapes as in test_gpu_ragged.py with the timeline on (JS_OPT_TRACE selects this kernel).
Widths that are not multiples of 8 (rows of symbols and noise that do not start on 16 bytes, padded rows of encodings), and
batches of several row tiles, out of which finished samples are moved."""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from parity import check_samples

pytestmark = pytest.mark.gpu

#         T    H                         batch  trace
SHAPES = [(129, (250, 127, 99, 131), 300, 0), (77, (130, 64, 65, 200), 131, 0), (9, (13, 9, 8, 7), 3, 0), (256, (256, 512, 256, 264), 290, 0),
          (129, (250, 127), 130, 1), (130, (385, 130), 300, 1), (200, (99,), 70, 1), (112, (128, 96), 257, 1)]


@pytest.mark.parametrize("T,H,batch,trace", SHAPES)
def test_grid_kernel(T, H, batch, trace):
    import __graft_entry__ as ge
    ge.build()
    import paper_2002_03629_b200 as p
    cfg = si.MadeConfig("ragged_grid", 67, D=T, C=1, H=H, act=si.ACT_GELU_TANH if T == 77 else si.ACT_RELU, prec=si.PREC_BF16, batch=batch,
                        noise_kind=si.NOISE_UNIFORM_ICDF if T == 200 else si.NOISE_LOGISTIC, w_var_scale=3.0, b_var=0.1)
    W, b = si.made_weights(cfg)
    lut, noise = si.made_lut(cfg), si.draw_noise(cfg)
    orc = oracle.from_config(cfg, W, b, lut)
    model = p.Model.from_config(cfg, W, b, lut)
    model.set_option(p.JS_OPT_TRACE, trace)
    d_noise = torch.from_numpy(noise).cuda()
    xstar = orc.sequential_batch(noise, cfg.noise_kind, threads=8)
    moved = 0
    for mode, block, init, compact in ((p.JS_JACOBI, 0, None, 1), (p.JS_JACOBI, 0, si.random_init(cfg, salt=1), 1), (p.JS_JACOBI, 0, None, 0),
                                       (p.JS_GS_JACOBI, max(1, T // 3), None, 1)):
        model.set_option(p.JS_OPT_COMPACT, compact)
        out = torch.full((batch, T), 255, dtype=torch.uint8, device="cuda")
        it = torch.full((batch,), -1, dtype=torch.int32, device="cuda")
        d_init = None if init is None else torch.from_numpy(init).cuda()
        assert p.jacobi_sample(model, d_noise, cfg.noise_kind, d_init, mode, block, 0, out, it) == 0
        st = model.stats()
        assert st.path == 0 and st.mma_flops > 0 and st.batch_iters_max == int(it.max())
        assert compact or st.compactions == 0
        moved += st.compactions
        audit = check_samples(orc, out.cpu().numpy(), xstar, noise, cfg.noise_kind)
        if mode == p.JS_JACOBI:
            clean = np.setdiff1d(np.arange(batch), audit["excused_samples"])[::7]
            want = np.array([orc.jacobi(noise[s], cfg.noise_kind, None if init is None else init[s])[1] for s in clean])
            np.testing.assert_array_equal(it.cpu().numpy()[clean], want)
    assert moved >= 1 or batch <= 256
    model.close()
