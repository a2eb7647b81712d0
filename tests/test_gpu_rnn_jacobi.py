"""Jacobi iterations and parameter gradients of the recurrent network on the tensor cores, where the kernels can go wrong: one and two
slots of 64 columns, several sequences in a unit and a ragged last unit, components around 16, 64 and 128, one and two chunks of
steps, all, half or a quarter of the columns per CTA, values that bf16 pieces cannot carry."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def reference(W, l, d, n, s0=None):
    W, l, d = W.double(), l.double(), d.double()
    s = torch.zeros_like(l) if s0 is None else s0.double()
    for _ in range(n):
        u = torch.zeros_like(l)
        u[:, :-1] = (d * s)[:, 1:]
        s = l + u @ W
    return s


def draw(B, T, H):
    g = torch.Generator("cuda").manual_seed(1000 * B + 10 * T + H)
    W = torch.randn((H, H), generator=g, device="cuda") * 0.1
    return W, torch.randn((B, T, H), generator=g, device="cuda"), torch.rand((B, T, H), generator=g, device="cuda"), torch.randn(
        (B, T, H), generator=g, device="cuda")


# fp32 multiply-adds in any order stay within sqrt(K) rounding steps of 2^-24 in the 2-norm, K <= 128 products: 7e-7
@pytest.mark.parametrize("B,T,H", [(1, 1, 4), (2, 2, 16), (1, 63, 20), (1, 64, 64), (1, 65, 68), (1, 80, 128), (3, 81, 112), (1, 128, 128),
                                   (150, 64, 64), (299, 64, 128), (297, 43, 36), (451, 32, 124), (500, 31, 8), (1500, 12, 32), (149, 65, 48)])
def test_against_64_bits(B, T, H):
    import paper_2002_03629_b200.rnn as rnn
    W, l, d, s0 = draw(B, T, H)
    for n, s in ((1, None), (2, None), (3, s0), (min(T, 9), None), (T + 1, s0)):
        got, want = rnn.rnn_bptt_jacobi(W, l, d, n, s0=s), reference(W, l, d, n, s)
        assert ((got.double() - want).norm() / want.norm()).item() < 7e-7, n


def plain(W, l, d, n, s0):
    """fp32 multiply-adds, component sums in ascending order."""
    W, l, d = W.cpu().numpy(), l.cpu().numpy(), d.cpu().numpy()
    s = np.zeros_like(l) if s0 is None else s0.cpu().numpy()
    with np.errstate(all="ignore"):
        for _ in range(n):
            new = l.copy()
            u = d * s
            for k in range(W.shape[0]):
                new[:, :-1] += u[:, 1:, k, None] * W[k]
            s = new
    return s


@pytest.mark.parametrize("T,H", [(20, 12), (70, 100)])
def test_values_beyond_the_pieces(T, H):
    """Infinities and NaN reach the steps that depend on them and no others; finite values that would round to an infinite bf16
    number stay finite; a start iterate's infinity is forgotten after T iterations."""
    import paper_2002_03629_b200.rnn as rnn
    B = 300
    W, l, d, s0 = draw(B, T, H)
    big = l.clone()
    big[3, T - 2, 1] = float("inf")
    big[4, 5, 2] = float("nan")
    big[200] *= 0
    big[200, T - 1, 0] = 3.4e38
    d[200] = 1.0
    for n, start in ((1, None), (4, None), (2, s0)):
        got, want = rnn.rnn_bptt_jacobi(W, big, d, n, s0=start).cpu().numpy(), plain(W, big, d, n, start)
        for i in (2, 3, 4, 5, 199, 200, 201, B - 1):
            np.testing.assert_array_equal(np.isfinite(got[i]), np.isfinite(want[i]))
            m = np.isfinite(want[i])
            scale = np.abs(want[i][m]).max()
            assert np.abs(got[i][m].astype(np.float64) - want[i][m]).max() <= 1e-5 * scale, (n, i)
    bad = s0.clone()
    bad[7, 2, 1] = float("inf")
    assert torch.equal(rnn.rnn_bptt_jacobi(W, l, d, T + 2, s0=bad)[:7], rnn.rnn_bptt_jacobi(W, l, d, T + 2)[:7])
    assert torch.isfinite(rnn.rnn_bptt_jacobi(W, l, d, T, s0=bad)).all()


def test_in_place():
    """The states may replace the direct gradients, the derivatives or the start iterate."""
    import paper_2002_03629_b200.rnn as rnn
    W, l, d, s0 = draw(155, 70, 64)
    want = rnn.rnn_bptt_jacobi(W, l, d, 6, s0=s0)
    for which in range(3):
        a = [l.clone(), d.clone(), s0.clone()]
        assert torch.equal(rnn.rnn_bptt_jacobi(W, a[0], a[1], 6, s0=a[2], out=a[which]), want)


@pytest.mark.parametrize("B,T,H,d_in", [(1, 25, 4, 1), (1, 64, 32, 3), (2, 65, 36, 4), (1, 128, 128, 16), (74, 48, 100, 1), (75, 66, 64, 5), (148, 63, 68, 2),
                                        (300, 127, 128, 1), (2, 24, 128, 2)])
def test_parameter_gradients_against_64_bits(B, T, H, d_in):
    import paper_2002_03629_b200.rnn as rnn
    _, s, d, h = draw(B, T, H)
    x = torch.rand((B, T, d_in), device="cuda")
    g = d.double() * s.double()
    want = torch.einsum("bti,btj->bij", g[:, 1:], h.double()[:, :-1]), torch.einsum("bti,btc->bic", g, x.double()), g.sum(1)
    for a, b in zip(rnn.rnn_param_grads(s, d, h, x), want):
        assert ((a.double() - b).norm() / b.norm()).item() < 7e-7
    # Factors of one sign, as a network's states are: the running sums are rounded towards zero, eight of them at most in an accumulator, each by
    # less than 2^-23 of its value at that time, which grows evenly to the whole (4.5 / 8 of it on average): 5e-7.
    g, hh = d.double() * s.abs().double(), h.abs()
    want = torch.einsum("bti,btj->bij", g[:, 1:], hh.double()[:, :-1])
    assert ((rnn.rnn_param_grads(s.abs(), d, hh, x)[0].double() - want).norm() / want.norm()).item() < 7e-7
    # a value that the pieces cannot carry: its sequence alone, the entries that it reaches alone
    s[0, T - 1, 1] = float("inf")
    h[0, 0, 2] = 3.39e38
    s[0, 1] = s[0, 1].abs() * 1e-30
    dWh, _, db = rnn.rnn_param_grads(s, d, h, x)
    g = d.double() * s.double()
    row = torch.arange(H, device="cuda") != 1
    want = torch.einsum("ti,tj->ij", g[0, 1:], h[0].double()[:-1])[row]
    assert torch.isfinite(dWh[0, row]).all() and not torch.isfinite(dWh[0, 1]).any() and not torch.isfinite(db[0, 1])
    assert ((dWh[0, row].double() - want).abs() <= 1e-5 * want.abs() + 1e-4).all()
    if B > 1:
        assert torch.isfinite(dWh[1:]).all()


@pytest.mark.parametrize("B,T,H", [(1, 25, 4), (2, 70, 128), (160, 40, 36)])
def test_parameter_gradients_beyond_fp32(B, T, H):
    """Finite operands whose products leave fp32 give what multiply-adds give: an infinity where one does, no NaN, and the sums that stay
    finite as they are."""
    import paper_2002_03629_b200.rnn as rnn
    _, s, d, h = draw(B, T, H)
    x = torch.zeros((B, T, 1), device="cuda")
    s, h = s.sign() + s, h.sign() + h
    d[:] = 1.0
    # (bf16 rounds 1.003e30 and 1.9e30 up and the others down: the products of their pieces leave fp32 with either sign)
    s[0, T - 2, 0], s[0, T - 2, 1] = 1.2345e30, 1.003e30
    h[0, T - 3, 2], h[0, T - 3, 3] = 1.9e30, -1.3e30
    got = rnn.rnn_param_grads(s, d, h, x)[0].cpu().numpy()
    g, hp = s.cpu().numpy(), h.cpu().numpy()
    with np.errstate(all="ignore"):
        want = sum(g[:, t, :, None] * hp[:, t - 1, None, :] for t in range(1, T))
    assert want[0, 1, 2] == np.inf and want[0, 1, 3] == -np.inf and not np.isnan(want).any()
    m = np.isfinite(want)
    np.testing.assert_array_equal(got[~m], want[~m])
    # T products of 24 bits, the largest of a sum being 2e30 and summed in any order: T rounding steps of 2^-24 of the absolute sum
    scale = sum(np.abs(g[:, t, :, None].astype(np.float64) * hp[:, t - 1, None, :]) for t in range(1, T))
    assert (np.abs(got[m].astype(np.float64) - want[m]) <= 2 * T * 2.0 ** -24 * scale[m]).all()


@pytest.mark.parametrize("scale", [2.0 ** -20, 2.0 ** -105, 2.0 ** -118])
@pytest.mark.parametrize("B,T,H", [(1, 33, 8), (2, 100, 128), (300, 30, 64)])
def test_small_values_keep_their_bits(B, T, H, scale):
    """States and operands near the lower end of fp32 are as exact as others, relative to their own size: 7e-7 in the 2-norm as above
    (at 2^-118 the smallest fp32 number, 2^-149, is below 2^-30 of the values' size and does not show)."""
    import paper_2002_03629_b200.rnn as rnn
    W, l, d, s0 = draw(B, T, H)
    l, s0 = l * scale, s0 * scale
    for n, s in ((2, None), (3, s0), (9, None)):
        got, want = rnn.rnn_bptt_jacobi(W, l, d, n, s0=s), reference(W, l, d, n, s)
        assert ((got.double() - want).norm() / want.norm()).item() < 7e-7, n
    # a component that hears of the others by small weights alone
    W2, l2 = W.clone(), l / scale
    W2[:, 1] *= scale
    l2[:, :, 1] = 0
    got, want = rnn.rnn_bptt_jacobi(W2, l2, d, 4)[:, :, 1].double(), reference(W2, l2, d, 4)[:, :, 1]
    assert ((got - want).norm() / want.norm().clamp_min(1e-300)).item() < 7e-7
    h, x = torch.rand((B, T, H), device="cuda"), torch.ones((B, T, 1), device="cuda")
    for g, hh in ((s0, h), (s0 / scale, h * scale)):
        want = torch.einsum("bti,btj->bij", (d.double() * g.double())[:, 1:], hh.double()[:, :-1])
        got = rnn.rnn_param_grads(g, d, hh, x)[0].double()
        assert ((got - want).norm() / want.norm()).item() < 7e-7


def test_more_than_two_to_the_31_steps():
    """A batch whose steps, let alone its values, no 32-bit number counts, in place (34 GB): the first and the last sequences, some around
    the 2^31st value and the 2^31st step from the end."""
    import paper_2002_03629_b200.rnn as rnn
    T, H = 128, 4
    B = 2 ** 31 // T + 300
    if torch.cuda.mem_get_info()[0] < 40 << 30:
        pytest.skip("needs 40 GB of device memory")
    g = torch.Generator("cuda").manual_seed(31)
    W = torch.randn((H, H), generator=g, device="cuda") * 0.1
    l = torch.empty((B, T, H), device="cuda").uniform_(0.25, 1.0, generator=g)       # the derivatives too: both are only read
    some = sorted({b for c in (0, 150, 300, B // 4, B // 2, B - 1) for b in range(c - 3, c + 4) if 0 <= b < B})
    before = l[some].clone()
    got = rnn.rnn_bptt_jacobi(W, l, l, 5, out=l)[some]
    want = reference(W, before, before, 5)
    assert ((got.double() - want).norm(dim=(1, 2)) / want.norm(dim=(1, 2))).max().item() < 7e-7


@pytest.mark.parametrize("B,T,H", [(1, 30, 8), (3, 100, 128), (400, 70, 64), (900, 30, 20)])
def test_waits_that_give_up(B, T, H):
    """Without any patience every block gives up at its first wait: all outputs are NaN, the status says why, and the calls that follow
    find shared and tensor memory as they need them.  With the usual patience the status stays as it was."""
    import paper_2002_03629_b200.rnn as rnn
    W, l, d, h = draw(B, T, H)
    x = torch.rand((B, T, 2), device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    s = rnn.rnn_bptt_jacobi(W, l, d, 5, status=status)
    grads = rnn.rnn_param_grads(s, d, h, x, status=status)
    assert int(status) == 0
    for _ in range(3):
        status.zero_()
        assert torch.isnan(rnn.rnn_bptt_jacobi(W, l, d, 5, status=status, wait_ns=0)).all() and int(status) == rnn.RNN_ERR_TIMEOUT
        status.zero_()
        for g in rnn.rnn_param_grads(s, d, h, x, status=status, wait_ns=0):
            assert torch.isnan(g).all()
        assert int(status) == rnn.RNN_ERR_TIMEOUT
        rnn.rnn_bptt_jacobi(W, l, d, 5, wait_ns=0)
        status.fill_(7)
        assert torch.equal(rnn.rnn_bptt_jacobi(W, l, d, 5, status=status), s)
        assert all(torch.equal(a, b) for a, b in zip(rnn.rnn_param_grads(s, d, h, x, status=status), grads))
        assert int(status) == 7
