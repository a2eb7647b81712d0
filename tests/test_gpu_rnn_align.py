"""The recurrent-network entry points take any fp32 pointer: views that start one to three floats off a 16-byte boundary
(parameters carved out of one flat buffer, say) give the very values of aligned tensors, in every form of the kernels
(one, two or more sequences per CTA; Jacobi iterations shared by clusters, thread groups, pairs, or one per CTA)."""
import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPES = [(64, 128, 1), (33, 36, 16), (12, 20, 5), (101, 128, 149), (120, 128, 150), (9, 8, 300), (8, 4, 460)]


def off(t, k):
    """A contiguous copy of t whose first element lies k floats behind a 16-byte boundary."""
    buf = torch.empty(t.numel() + 4, device=t.device)
    v = buf[k:k + t.numel()].view(t.shape)
    v.copy_(t)
    assert v.is_contiguous() and v.data_ptr() % 16 == 4 * k
    return v


@pytest.mark.parametrize("T,H,B", SHAPES)
def test_views_at_any_float(T, H, B):
    import paper_2002_03629_b200.rnn as rnn
    g = torch.Generator("cuda").manual_seed(T + H + B)

    def rand(*shape):
        return torch.randn(shape, generator=g, device="cuda") * 0.1
    ins = [rand(H, H), rand(H, 2), rand(H), rand(3, H), rand(3), rand(B, T, 2), rand(B, T, 3)]
    want = rnn.rnn_forward(*ins)
    h, d, l, _ = want
    seq = rnn.rnn_bptt_sequential(ins[0], l, d)
    jac = rnn.rnn_bptt_jacobi(ins[0], l, d, 4, s0=seq)
    grads = rnn.rnn_param_grads(seq, d, h, ins[5])
    for k in (1, 2, 3):
        moved = [off(t, k) for t in ins]
        for which in (*range(len(ins)), None):           # one argument at a time, then all of them
            args = [m if which in (i, None) else t for i, (m, t) in enumerate(zip(moved, ins))]
            for a, b in zip(rnn.rnn_forward(*args), want):
                assert torch.equal(a, b)
        out = torch.zeros_like(l)
        for w, dd, ll, o in ((moved[0], d, l, out), (ins[0], off(d, k), l, out), (ins[0], d, off(l, k), out), (ins[0], d, l, off(out, k))):
            assert torch.equal(rnn.rnn_bptt_sequential(w, ll, dd, out=o), seq)
            assert torch.equal(rnn.rnn_bptt_jacobi(w, ll, dd, 4, s0=off(seq, k), out=o), jac)
        for i in range(4):
            args = [off(t, k) if i == j else t for j, t in enumerate((seq, d, h, ins[5]))]
            for a, b in zip(rnn.rnn_param_grads(*args), grads):
                assert torch.equal(a, b)


def test_outputs_of_the_c_entry_points_at_any_float():
    """The binding allocates the outputs of the forward pass and of the gradients; a C caller places them anywhere."""
    import ctypes as C
    import paper_2002_03629_b200.rnn as rnn
    lib = rnn._lib()
    T, H, B = 10, 12, 3
    g = torch.Generator("cuda").manual_seed(1)

    def rand(*shape):
        return torch.randn(shape, generator=g, device="cuda") * 0.1
    ins = [rand(H, H), rand(H, 1), rand(H), rand(1, H), rand(1), rand(B, T, 1), rand(B, T, 1)]
    want = rnn.rnn_forward(*ins)
    seq = rnn.rnn_bptt_sequential(ins[0], want[2], want[1])
    grads = rnn.rnn_param_grads(seq, want[1], want[0], ins[5])
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    ptr = lambda t: C.c_void_p(t.data_ptr())
    for which in range(4):
        outs = [off(torch.zeros_like(t), 1 if i == which else 0) for i, t in enumerate(want)]
        assert lib.rnn_forward(*map(ptr, ins), B, T, H, 1, 1, *map(ptr, outs), stream) == 0
        assert all(torch.equal(a, b) for a, b in zip(outs, want))
    for which in range(3):
        outs = [off(torch.zeros_like(t), 1 if i == which else 0) for i, t in enumerate(grads)]
        assert lib.rnn_param_grads(ptr(seq), ptr(want[1]), ptr(want[0]), ptr(ins[5]), B, T, H, 1, *map(ptr, outs), stream) == 0
        assert all(torch.equal(a, b) for a, b in zip(outs, grads))
