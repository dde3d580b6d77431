"""The tensor-core kernel for a batch of tokens and for prompts on small layers, against the CPU oracle, on a B200: edges of its
token blocks (16 to 64 wide, one or several), of the 128-channel super-blocks and of its 128-k steps, with and without a K split,
with two and with three groups of unpacking warps.  Some of the calls are near a line of the dispatch; test_routes_gpu.py runs all of them on
this kernel."""
import numpy as np
import pytest

from oracle import qlinear_oracle as O
from workloads import configs as C

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P(_built_library):
    import paper_2505_00232_b200 as P
    return P


@pytest.fixture(scope="module")
def torch():
    import torch
    assert torch.cuda.is_available(), "these tests need a CUDA device"
    return torch


def spec(N, K, bits, group):
    return C.LayerSpec("t", N, K, bits, group, *((-8, 7) if bits == 4 else (-128, 127)))


def check(P, torch, N, K, bits, group, M, rows, act="silu"):
    """One layer, two layers in one launch (of different widths), the gated pair; the oracle on `rows` of the outputs."""
    specs = [spec(n, K, bits, group) for n in (N, N, N + 136)]
    w = [C.layer_weights(9100 + M + N + K + i, s) for i, s in enumerate(specs)]
    x = C.layer_activations(9100 + M, specs[0], M)
    lins = [P.QLinear.from_weights(q, s, bits, group, device="cuda:0") for q, s in w]
    xd = torch.from_numpy(x).cuda()
    buf = torch.full((M + 2, N), 7.0, dtype=torch.float16, device="cuda")
    one = lins[0].forward(xd, out=buf[1:M + 1])
    many = P.qlinear_forward_group([lins[0], lins[2]], xd)
    gated = P.qlinear_forward_gated(lins[0], lins[1], xd, act)
    torch.cuda.synchronize()
    assert lins[0].device_status() == (0, 0)
    assert (buf[0] == 7).all() and (buf[M + 1] == 7).all()
    for y, (q, s) in zip((one, *many), (w[0], w[0], w[2])):
        y64, A, _ = O.linear(x, q[rows], s[rows], group)
        ok, rel, worst = O.check_against(y.cpu().numpy()[:, rows], y64, A)
        assert ok, (rel, worst)
    g64, bound, _ = O.gated_linear(x, w[0][0][rows], w[0][1][rows], w[1][0][rows], w[1][1][rows], group, act)
    ok, rel, worst = O.check_gated(gated.cpu().numpy()[:, rows], g64, bound)
    assert ok, (rel, worst)
    again = torch.empty_like(gated)
    for _ in range(3):                                                   # run-to-run identical
        P.qlinear_forward_gated(lins[0], lins[1], xd, act, out=again)
        assert torch.equal(gated, again) and torch.equal(one, lins[0].forward(xd))


SMALL = [(N, K, bits, group, M) for N, K in ((8, 160), (136, 352), (264, 1024), (640, 1152)) for M in (65, 96, 97, 128, 129, 300)
         for bits, group in ((4, 32), (4, 0), (8, 0))]
LARGE = [(2304, 3776, 4, 32, 25), (2304, 4032, 4, 0, 32), (2312, 3712, 8, 0, 31), (2304, 9216, 4, 32, 17), (4096, 12544, 4, 32, 9),
         (4104, 12576, 8, 0, 16), (1024, 4096, 4, 32, 33), (1032, 4000, 8, 0, 48), (1032, 1664, 4, 128, 49), (1032, 1568, 8, 0, 64), (14336, 1024, 4, 32, 64)]


@pytest.mark.parametrize("N,K,bits,group,M", SMALL)
def test_small_layers(P, torch, N, K, bits, group, M):
    """Several token blocks; K with a last half step (352 and 1152 are odd in 64 k), with 32 k of it (160, 352), a K split."""
    check(P, torch, N, K, bits, group, M, np.arange(N), "gelu_tanh" if M == 97 else "silu")


@pytest.mark.parametrize("N,K,bits,group,M", LARGE)
def test_large_layers_of_the_batch_stage(P, torch, N, K, bits, group, M):
    """Up to 64 tokens, layers large enough for this kernel or nearly so; int4 up to 32 tokens: three groups."""
    check(P, torch, N, K, bits, group, M, np.r_[0:64, N - 72:N])


def test_calls_on_two_streams_do_not_meet(P, torch):
    """No scratch is shared: two layers split along K, on streams that are not ordered against each other."""
    layers = [spec(1024, 8192, 4, 32), spec(1024, 8192, 8, 0)]
    lins = [P.QLinear.from_weights(*C.layer_weights(9700 + i, s), s.bits, s.group, device="cuda:0") for i, s in enumerate(layers)]
    xs = [torch.from_numpy(C.layer_activations(9700 + i, s, 100)).cuda() for i, s in enumerate(layers)]
    first = [l.forward(x) for l, x in zip(lins, xs)]
    outs = [torch.empty_like(f) for f in first]
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    for _ in range(50):
        for l, x, o, st in zip(lins, xs, outs, streams):
            l.forward(x, out=o, stream=st)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(first, outs)) and lins[0].device_status() == (0, 0)
