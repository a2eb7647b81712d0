"""The cluster kernel of small fp32 masked MLPs at the edges of its tiles: one unit, widths around the 32 outputs of a
warp and the 16 inputs of a product step, every cluster size, one sample, batches that leave the last cluster ragged."""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from oracle import Oracle
from parity import check_samples

pytestmark = pytest.mark.gpu

#        T    H            batch   (cluster size grows with the widest layer: 1, 2, 4, 8 CTAs)
SHAPES = [(2, (1,), 1), (16, (17, 33), 8), (33, (96,), 150), (97, (31, 97), 5), (130, (193,), 70), (63, (385, 8), 33),
          (257, (200, 120), 300)]


def _pkg():
    import __graft_entry__ as ge
    ge.build()
    import paper_2002_03629_b200 as p
    return p


@pytest.mark.parametrize("T,H,batch", SHAPES)
@pytest.mark.parametrize("skip", [1, 0])
def test_binary(T, H, batch, skip):
    p = _pkg()
    cfg = si.MadeConfig("small", 61, D=T, C=1, H=H, act=si.ACT_GELU_TANH if T == 63 else si.ACT_RELU, prec=si.PREC_F32,
                        batch=batch, noise_kind=si.NOISE_LOGISTIC if T % 2 else si.NOISE_UNIFORM_ICDF, w_var_scale=4.0, b_var=0.1)
    W, b = si.made_weights(cfg)
    lut, noise = si.made_lut(cfg), si.draw_noise(cfg)
    orc = oracle.from_config(cfg, W, b, lut)
    model = p.Model.from_config(cfg, W, b, lut)
    model.set_option(p.JS_OPT_FRONTIER_SKIP, skip)
    xstar = orc.sequential_batch(noise, cfg.noise_kind, threads=8)
    for init in (None, si.random_init(cfg, salt=2)):
        out = torch.full((batch, T), 255, dtype=torch.uint8, device="cuda")
        it = torch.full((batch,), -1, dtype=torch.int32, device="cuda")
        d_init = None if init is None else torch.from_numpy(init).cuda()
        rc = p.jacobi_sample(model, torch.from_numpy(noise).cuda(), cfg.noise_kind, d_init, p.JS_JACOBI, 0, 0, out, it)
        st = model.stats()
        assert rc == 0 and st.path == 1 and st.batch_iters_max == int(it.max())
        audit = check_samples(orc, out.cpu().numpy(), xstar, noise, cfg.noise_kind)
        want = np.array([orc.jacobi(noise[s], cfg.noise_kind, None if init is None else init[s])[1] for s in range(batch)])
        clean = np.setdiff1d(np.arange(batch), audit["excused_samples"])
        np.testing.assert_array_equal(it.cpu().numpy()[clean], want[clean])
    out = torch.empty((batch, T), dtype=torch.uint8, device="cuda")
    if int(want.max()) > 2:
        assert p.jacobi_sample(model, torch.from_numpy(noise).cuda(), cfg.noise_kind, None, p.JS_JACOBI, 0, 1, out) == p.JS_NOT_CONVERGED
    model.close()


@pytest.mark.parametrize("T,H,batch", SHAPES)
def test_continuous(T, H, batch):
    """eps = 0 returns the very floats of the strict order, which another kernel computes with the same arithmetic."""
    p = _pkg()
    cfg = si.MadeConfig("small_real", 62, D=T, C=2, H=H, act=si.ACT_RELU, prec=si.PREC_F32, batch=batch,
                        noise_kind=si.NOISE_LOGISTIC, w_var_scale=2.0, b_var=0.05)
    W, b = si.made_real_weights(cfg)
    lut = np.zeros(2, np.float32)
    model = p.Model.made(T, 2, list(H), cfg.act, cfg.prec, W, b, lut, batch)
    noise = torch.from_numpy(si.draw_noise(cfg)).cuda()
    seq, x = (torch.full((batch, T), 7.0, device="cuda") for _ in range(2))
    assert p.sequential_sample_real(model, noise, seq) == 0
    assert p.jacobi_sample_real(model, noise, None, p.JS_JACOBI, 0, 0, 0.0, x) == 0
    assert torch.equal(seq, x)
    orc = Oracle.made(T, 2, list(H), cfg.act, cfg.prec, W, b, lut)
    ref = np.stack([orc.sequential_real(noise[s].cpu().numpy()) for s in range(min(batch, 4))])
    err = np.abs(seq[:4].cpu().numpy() - ref) / np.maximum(1.0, np.abs(ref))
    assert err.max() <= 5e-4          # the fp32 bound of the other tests of continuous states
    model.close()
