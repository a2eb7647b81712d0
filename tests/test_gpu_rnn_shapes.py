"""Every form of the recurrent-network kernels at the edges of its range: sequences per CTA (1, 2, 4) with a ragged last
CTA, Jacobi iterations shared by a cluster of 8 or 4 CTAs, by thread groups of one CTA, by a pair of sequences, or one
sequence per CTA; steps and widths around the tiles.  Tolerance as in test_gpu_rnn.py (fp32 sums of at most 130 products)."""
import numpy as np
import pytest
import torch

import synth_inputs as si
from oracle import rnn_oracle as ro
from test_gpu_rnn import close, dev

pytestmark = pytest.mark.gpu

#          T    H   d_in d_out B
SHAPES = [(64, 128, 1, 1, 1), (65, 36, 2, 3, 15), (32, 128, 1, 1, 16), (127, 124, 16, 16, 5), (100, 128, 1, 1, 66), (31, 128, 1, 2, 4),
          (31, 8, 1, 1, 148), (101, 128, 1, 1, 149), (104, 128, 3, 1, 151), (128, 128, 1, 1, 150), (7, 4, 1, 1, 297), (17, 132 - 4, 1, 1, 299)]


@pytest.mark.parametrize("T,H,d_in,d_out,B", SHAPES)
def test_shapes(T, H, d_in, d_out, B):
    import paper_2002_03629_b200.rnn as rnn
    cfg = si.RnnConfig("shape", 21, T=T, H=H, d_in=d_in, d_out=d_out, batch=B)
    Wh, Wx, b, Wo, bo = si.rnn_weights(cfg)
    rng = np.random.default_rng(T * H + B)
    b, bo = (rng.normal(0, 0.1, v.shape).astype(np.float32) for v in (b, bo))
    x, r = si.rnn_sequences(cfg)
    W, (dx, dr) = dev(Wh, Wx, b, Wo, bo), dev(x, r)
    h, d, l, loss = rnn.rnn_forward(*W, dx, dr)
    seqs = sorted({0, 1 % B, B // 2, B - 1})
    want = {i: ro.forward(Wh, Wx, b, Wo, bo, x[i], r[i]) for i in seqs}
    for i in seqs:
        for name, got in (("h", h), ("d", d), ("l", l)):
            close(got[i], want[i][name], f"{name}[{i}]")
        close(loss[i], np.float64(want[i]["loss"]), f"loss[{i}]")
    s0 = torch.from_numpy(rng.normal(size=(B, T, H)).astype(np.float32)).cuda()
    ln, dn, s0n = (v.cpu().double().numpy() for v in (l, d, s0))
    seq = rnn.rnn_bptt_sequential(W[0], l, d)
    for i in seqs:
        close(seq[i], ro.backprop_exact(Wh, ln[i], dn[i]), f"sequential[{i}]")
    for n in (1, 4, T - 1, T + 2):
        a, a0 = rnn.rnn_bptt_jacobi(W[0], l, d, n), rnn.rnn_bptt_jacobi(W[0], l, d, n, s0=s0)
        for i in seqs:
            close(a[i], ro.backprop_jacobi(Wh, ln[i], dn[i], n), f"jacobi_{n}[{i}]")
            close(a0[i], ro.backprop_jacobi(Wh, ln[i], dn[i], n, s0n[i]), f"jacobi_{n} from s0[{i}]")
    dWh, dWx, db = rnn.rnn_param_grads(seq, d, h, dx)
    hn, sn = h.cpu().double().numpy(), seq.cpu().double().numpy()
    for i in seqs:
        g = ro.param_grads(sn[i], dn[i], hn[i], x[i])
        close(dWh[i], g[0], f"dWh[{i}]")
        close(dWx[i], g[1], f"dWx[{i}]")
        close(db[i], g[2], f"db[{i}]")


# one to four sequences per CTA, with outputs and inputs whose sums go one, two or four at a time, and what is left of them
@pytest.mark.parametrize("d_in,d_out,B", [(1, 1, 3), (5, 1, 3), (4, 2, 3), (2, 3, 2), (3, 7, 150), (1, 4, 299), (6, 5, 445), (16, 16, 593)])
def test_forward_with_many_outputs(d_in, d_out, B):
    import paper_2002_03629_b200.rnn as rnn
    cfg = si.RnnConfig("shape", 22, T=9, H=20, d_in=d_in, d_out=d_out, batch=B)
    Wh, Wx, b, Wo, bo = si.rnn_weights(cfg)
    rng = np.random.default_rng(B)
    b, bo = (rng.normal(0, 0.1, v.shape).astype(np.float32) for v in (b, bo))
    x, r = rng.normal(size=(B, 9, d_in)).astype(np.float32), rng.normal(size=(B, 9, d_out)).astype(np.float32)
    h, d, l, loss = rnn.rnn_forward(*dev(Wh, Wx, b, Wo, bo, x, r))
    for i in sorted({0, 1, B // 2, B - 2, B - 1}):
        want = ro.forward(Wh, Wx, b, Wo, bo, x[i], r[i])
        for name, got in (("h", h), ("d", d), ("l", l)):
            close(got[i], want[name], f"{name}[{i}]")
        close(loss[i], np.float64(want["loss"]), f"loss[{i}]")


# rounds of sequences per SM: three (one per CTA), two and four (pairs), the last of them ragged
@pytest.mark.parametrize("T,H,B", [(37, 64, 297), (37, 64, 296), (101, 128, 443), (101, 128, 445)])
def test_rounds_of_sequences(T, H, B):
    import paper_2002_03629_b200.rnn as rnn
    g = torch.Generator("cuda").manual_seed(B)
    Wh = torch.randn((H, H), generator=g, device="cuda") * 0.1
    l, d = torch.randn((B, T, H), generator=g, device="cuda"), torch.rand((B, T, H), generator=g, device="cuda")
    a = rnn.rnn_bptt_jacobi(Wh, l, d, 6)
    ln, dn, W = l.cpu().double().numpy(), d.cpu().double().numpy(), Wh.cpu().numpy()
    for i in sorted({0, 147, 148, B // 2, B - 2, B - 1}):
        close(a[i], ro.backprop_jacobi(W, ln[i], dn[i], 6), f"jacobi[{i}]")
