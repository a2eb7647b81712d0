"""The cluster kernel with more samples than one round of clusters holds, with a ragged last cluster, and with the widest weight share
that it takes.  A sample's sums depend neither on the cluster that it falls to nor on how many samples share it, so every row of a large
batch has to be the row that a batch of a few samples gives (whose agreement with the oracle test_gpu_cluster.py checks), bit for
bit, in every call."""
import pytest
import torch

import synth_inputs as si

pytestmark = pytest.mark.gpu


def make(T, H, batch):
    import __graft_entry__ as ge
    ge.build()
    import paper_2002_03629_b200 as p
    cfg = si.MadeConfig("rounds", 73, D=T, C=1, H=H, act=si.ACT_RELU, prec=si.PREC_BF16, batch=batch, noise_kind=si.NOISE_LOGISTIC, w_var_scale=1.0, b_var=0.1)
    W, b = si.made_weights(cfg)
    return p, cfg, p.Model.from_config(cfg, W, b, si.made_lut(cfg)), torch.from_numpy(si.draw_noise(cfg)).cuda()


def by_the_cluster_kernel(model):
    """After a Jacobi call of several passes: the grid-wide kernel skips final tiles, the cluster kernel computes every tile in every pass."""
    s = model.stats()
    assert s.path == 0 and s.iterations >= 2
    return s.tiles_skipped == 0


# Samples a cluster, clusters, two rounds?  24, 19 (of 8 CTAs, 148 SMs hold 18 at most), yes; 64, 40 (of 4 CTAs; 37), yes; 16, 19, yes; 8, 3, no.
# The last clusters hold 18, 4, 12 and 1.
@pytest.mark.parametrize("T,H,batch", [(784, (1024, 1024), 450), (200, (500,), 2500), (1024, (1536, 1536), 300), (1936, (2048, 2048, 2048), 17)])
def test_rounds(T, H, batch):
    p, cfg, model, noise = make(T, H, batch)
    few = 8
    iters = torch.empty(batch, dtype=torch.int32, device="cuda")
    for mode, block in ((p.JS_JACOBI, 0), (p.JS_GS_JACOBI, T // 4)):
        want, want_it = torch.empty((batch, T), dtype=torch.uint8, device="cuda"), torch.empty_like(iters)
        for lo in range(0, batch, few):
            hi = min(batch, lo + few)
            o, i = torch.empty((hi - lo, T), dtype=torch.uint8, device="cuda"), torch.empty(hi - lo, dtype=torch.int32, device="cuda")
            assert p.jacobi_sample(model, noise[lo:hi].clone(), cfg.noise_kind, None, mode, block, 0, o, i) == 0
            want[lo:hi], want_it[lo:hi] = o, i
        for _ in range(3):
            out = torch.full((batch, T), 7, dtype=torch.uint8, device="cuda")
            iters.fill_(-1)
            assert p.jacobi_sample(model, noise, cfg.noise_kind, None, mode, block, 0, out, iters) == 0
            if mode == p.JS_JACOBI:
                assert by_the_cluster_kernel(model)
            assert torch.equal(out, want) and torch.equal(iters, want_it)
    model.close()


# 16 samples a cluster leave the ring two loads, 8 samples more.
@pytest.mark.parametrize("T,H,batch,cluster", [(1296, (2048, 2048), 200, False), (1296, (2048, 2048), 100, True), (1296, (1024, 1600, 1750), 200, True),
                                               (1156, (2048, 2048), 200, True), (1024, (2048, 2048), 200, True)])
def test_short_rings(T, H, batch, cluster):
    p, cfg, model, noise = make(T, H, batch)
    out = torch.empty((batch, T), dtype=torch.uint8, device="cuda")
    assert p.jacobi_sample(model, noise, cfg.noise_kind, None, p.JS_JACOBI, 0, 0, out) == 0
    assert by_the_cluster_kernel(model) == cluster
    # noise one float off a 16-byte boundary: the cluster kernel in any case, the same samples (the other kernel sums in another order, which may
    # move a decision that nearly ties and with it the rest of that sample)
    off = torch.empty(noise.numel() + 4, device="cuda")[1:1 + noise.numel()].view(noise.shape)
    off.copy_(noise)
    out2 = torch.empty_like(out)
    assert p.jacobi_sample(model, off, cfg.noise_kind, None, p.JS_JACOBI, 0, 0, out2) == 0
    assert by_the_cluster_kernel(model)
    assert torch.equal(out, out2) if cluster else int((out == out2).all(1).sum()) >= batch - batch // 8
    model.close()
