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


def run_into(p, model, noise, nk, out, it, mode=0, block=0):
    """The C entry point with outputs anywhere that the device can write (mapped host memory here)."""
    import ctypes as C
    lib = p.load_library()
    ptr = lambda t: C.c_void_p(t.data_ptr())
    return lib.jacobi_sample(model._h, out.shape[0], ptr(noise), nk, None, mode, block, 0, ptr(out), ptr(it), C.c_void_p(torch.cuda.current_stream().cuda_stream))


@pytest.mark.parametrize("T,H,batch,prec,mode,block", [(16, (64,), 8, si.PREC_F32, 0, 0), (96, (128, 128), 64, si.PREC_BF16, 0, 0),
                                                       (96, (128, 128), 64, si.PREC_BF16, 2, 32), (96, (128,), 33, si.PREC_F32, 2, 32)])
def test_outputs_in_host_memory_are_complete_on_return(T, H, batch, prec, mode, block):
    """Small models' cluster kernels report with a fence that covers device memory; for outputs that the host reads
    directly the call has to wait for the stream."""
    p, cfg, model, noise = binary_model(T, H, batch, prec)
    ref = torch.zeros((batch, T), dtype=torch.uint8, device="cuda")
    it_ref = torch.zeros(batch, dtype=torch.int32, device="cuda")
    assert p.jacobi_sample(model, noise, cfg.noise_kind, None, mode, block, 0, ref, it_ref) == 0
    ref, it_ref = ref.cpu(), it_ref.cpu()
    out = torch.zeros((batch, T), dtype=torch.uint8).pin_memory()
    it = torch.zeros(batch, dtype=torch.int32).pin_memory()
    for _ in range(100):
        out.zero_()
        it.zero_()
        torch.cuda.synchronize()
        rc = run_into(p, model, noise, cfg.noise_kind, out, it, mode, block)
        over = torch.cuda.current_stream().query()
        assert rc == 0 and over
        assert torch.equal(out, ref) and torch.equal(it, it_ref)
    model.close()


def test_a_program_that_asked_for_blocking_waits_gets_them():
    """cudaDeviceScheduleBlockingSync: the calling thread sleeps while the GPU works (a spinning wait uses the whole core)."""
    import os
    import subprocess
    import sys
    code = """
import ctypes, time
cu = ctypes.CDLL("libcuda.so.1")
assert cu.cuInit(0) == 0 and cu.cuDevicePrimaryCtxSetFlags_v2(0, 4) == 0
import numpy as np
import torch
torch.cuda.init()
import paper_2002_03629_b200 as p, synth_inputs as si
cfg = si.MadeConfig("block", 72, D=400, C=2, H=(512,), act=si.ACT_RELU, prec=si.PREC_F32, batch=64, noise_kind=si.NOISE_LOGISTIC, w_var_scale=2.0, b_var=0.05)
W, b = si.made_real_weights(cfg)
m = p.Model.made(400, 2, [512], cfg.act, cfg.prec, W, b, np.zeros(2, np.float32), 64)
noise = torch.from_numpy(si.draw_noise(cfg)).cuda()
x = torch.empty((64, 400), device="cuda")
p.sequential_sample_real(m, noise, x)
torch.cuda.synchronize()
cpu, wall = time.thread_time(), time.perf_counter()
for _ in range(20):
    p.sequential_sample_real(m, noise, x)
cpu, wall = time.thread_time() - cpu, time.perf_counter() - wall
print("cpu", cpu, "wall", wall)
assert wall > 0.02 and cpu < 0.5 * wall, (cpu, wall)
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    run = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stdout + run.stderr


@pytest.mark.parametrize("T,H,batch", [(100, (512, 512), 64), (100, (96,), 8)])
def test_weights_that_do_not_come_end_the_call(T, H, batch):
    """Small fp32 models: no wait at all is allowed, so the CTAs' weights (up to 190 KB each) are not there at the first look.
    Whichever CTA of a cluster gives up, the call says so, and the model works afterwards, also on the kernel with grid barriers."""
    p, cfg, model, noise = binary_model(T, H, batch, si.PREC_F32)
    ref = torch.zeros((batch, T), dtype=torch.uint8, device="cuda")
    assert p.sequential_sample(model, noise, cfg.noise_kind, ref) == 0
    out = torch.zeros_like(ref)
    for _ in range(3):
        model.set_option(p.JS_OPT_SPIN_LIMIT, 0)
        try:
            rc = p.jacobi_sample(model, noise, cfg.noise_kind, None, p.JS_JACOBI, 0, 0, out)
        except p.JsError as e:
            assert e.code == p.JS_ERR_TIMEOUT
        else:                                            # (the weights may be there all the same where they are few)
            assert rc == 0 and len(H) == 1 and torch.equal(out, ref)
        model.set_option(p.JS_OPT_SPIN_LIMIT, 1 << 22)
        assert p.jacobi_sample(model, noise, cfg.noise_kind, None, p.JS_GS_JACOBI, 32, 0, out) == 0 and torch.equal(out, ref)
        out.zero_()
        assert p.jacobi_sample(model, noise, cfg.noise_kind, None, p.JS_JACOBI, 0, 0, out) == 0 and torch.equal(out, ref)
    model.close()
