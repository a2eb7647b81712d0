"""What a call has written when it returns: the calls end when the host sees a word that the last kernel writes, so the
outputs must be complete behind that word, for work on any stream."""
import numpy as np
import pytest
import torch

import synth_inputs as si

pytestmark = pytest.mark.gpu


def binary_model(T=96, H=(128, 128), batch=64, prec=si.PREC_BF16):
    import paper_2002_03629_b200 as p
    cfg = si.MadeConfig("reports", 71, D=T, C=1, H=H, act=si.ACT_RELU, prec=prec, batch=batch, noise_kind=si.NOISE_LOGISTIC, w_var_scale=3.0, b_var=0.1)
    W, b = si.made_weights(cfg)
    return p, cfg, p.Model.from_config(cfg, W, b, si.made_lut(cfg)), torch.from_numpy(si.draw_noise(cfg)).cuda()


def test_jacobi_gs_counts_are_there_for_another_stream():
    p, cfg, model, noise = binary_model()
    out = torch.zeros((cfg.batch, cfg.D), dtype=torch.uint8, device="cuda")
    it = torch.zeros(cfg.batch, dtype=torch.int32, device="cuda")
    assert p.jacobi_sample(model, noise, cfg.noise_kind, None, p.JS_JACOBI_GS, 16, 0, out, it) == 0
    torch.cuda.synchronize()
    want_x, want_it = out.cpu().numpy(), it.cpu().numpy()
    assert want_it.min() >= 1
    other = torch.cuda.Stream()
    for _ in range(200):
        it.zero_()
        out.zero_()
        torch.cuda.synchronize()
        assert p.jacobi_sample(model, noise, cfg.noise_kind, None, p.JS_JACOBI_GS, 16, 0, out, it) == 0
        with torch.cuda.stream(other):                   # ordered behind nothing but the call's return
            got_it, got_x = it.clone(), out.clone()
        np.testing.assert_array_equal(got_it.cpu().numpy(), want_it)
        np.testing.assert_array_equal(got_x.cpu().numpy(), want_x)
    model.close()


def test_jacobi_gs_leaves_nothing_queued_after_an_error():
    """A wait that gives up ends the call with launches of the same iteration behind it: they are over when it returns."""
    p, cfg, model, noise = binary_model()
    out = torch.zeros((cfg.batch, cfg.D), dtype=torch.uint8, device="cuda")
    it = torch.full((cfg.batch,), -7, dtype=torch.int32, device="cuda")
    model.set_option(p.JS_OPT_SPIN_LIMIT, 0)
    for _ in range(3):
        with pytest.raises(p.JsError) as e:
            p.jacobi_sample(model, noise, cfg.noise_kind, None, p.JS_JACOBI_GS, 16, 0, out, it)
        assert e.value.code == p.JS_ERR_TIMEOUT
        assert torch.cuda.current_stream().query()
    assert int((it != -7).sum()) == 0
    model.set_option(p.JS_OPT_SPIN_LIMIT, 1 << 22)
    assert p.jacobi_sample(model, noise, cfg.noise_kind, None, p.JS_JACOBI_GS, 16, 0, out, it) == 0
    ref = torch.zeros_like(out)
    assert p.sequential_sample(model, noise, cfg.noise_kind, ref) == 0
    assert torch.equal(out, ref) and int(it.min()) >= 1
    model.close()
