"""Plans of the CTA-pair prefill kernel that divide a launch more finely than blocks of 256 tokens: narrower blocks, K parts, and gated pairs
with fewer positions of 256 tokens than CTA pairs.  Which plan a call gets is checked without a device."""
import ctypes

import numpy as np
import pytest

from oracle import qlinear_oracle as O
from workloads import configs as C

SMS = 148
PAIR_TA = 6
# (tokens, channels, K, bits, group, width, parts): remainders in tokens, channels, k; the last block nearly empty
PLAIN = [(300, 2304, 9216, 4, 32, 160, 4), (257, 2800, 8224, 8, 0, 96, 2), (641, 4096, 2176, 4, 0, 192, 1), (1409, 2560, 1152, 4, 128, 224, 1), (1030, 4864, 1152, 8, 0, 160, 1)]
GATED = [(300, 8400, 1088, 4, 32, 160), (240, 17352, 960, 8, 0, 128), (168, 16640, 448, 8, 0, 96), (259, 13312, 1088, 4, 0, 160)]
GATED_ON_NARROW = [(330, 6144, 1120, 8, 0), (130, 9216, 1120, 8, 0)]      # (us, gemm_narrow.cuh / two accumulators: 16.1 / 18.1, 14.1 / 17.2)
# Two accumulators (the position's second one, at blocks of 160, 128, 96 and 64): one round and two, one k-step to many, few channels, the three activations
TWO_ACCUMULATORS = [(240, 17352, 960, 8, 0, 128, "gelu_tanh"), (161, 17152, 384, 4, 32, 96, "identity"), (391, 9216, 192, 4, 32, 160, "gelu_tanh"), (183, 17664, 128, 4, 32, 96, "silu"),
                    (415, 7424, 128, 8, 0, 160, "identity"), (1518, 1792, 1984, 4, 32, 160, "gelu_tanh"), (1100, 504, 224, 8, 0, 96, "silu"), (2000, 248, 32, 8, 0, 96, "gelu_tanh"),
                    (1029, 248, 160, 8, 0, 64, "identity"), (184, 256, 32, 8, 0, 32, "silu"), (228, 10752, 192, 4, 0, 128, "silu")]
# integer form: one pair of row super-blocks to many, one k-step to many, parts and narrow blocks
A8 = [(129, 256, 128, 4), (130, 200, 8192, 8), (200, 1024, 4096, 4), (333, 2296, 9216, 8), (700, 1024, 2304, 4), (1030, 4096, 1152, 8), (641, 9216, 256, 4)]

# and with its plan (tokens per tile, K parts, token blocks): int4 in 4 parts, remainders in tokens and channels
A8_PARTS = [((150, 256, 8192, 4), (32, 4, 5)), ((333, 504, 9216, 4), (64, 4, 6)), ((129, 2296, 8192, 4), (96, 4, 2)), ((257, 1000, 9216, 8), (96, 4, 3)), ((200, 1024, 14336, 4), (64, 4, 4)),
            ((200, 1024, 4096, 4), (64, 2, 4)), ((1030, 4096, 1152, 8), (128, 1, 9))]
# int8-activation decode: CTAs, CTAs per cluster
A8_DECODE = [((1, 1024, 4096, 8, 0), (128, 2)), ((2, 4096, 14336, 4, 0), (256, 1)), ((8, 2304, 9216, 4, 32), (288, 2)), ((7, 2304, 9216, 8, 0), (288, 2)), ((8, 1024, 4096, 4, 0), (128, 2)),
             ((1, 4096, 14336, 8, 0), (512, 2)), ((1, 256, 4096, 8, 0), (64, 4)), ((3, 264, 14336, 4, 32), (119, 7)), ((8, 64, 16384, 8, 0), (32, 8)), ((1, 14336, 4096, 4, 0), (448, 1))]


@pytest.fixture(scope="module")
def P(_built_library):
    import paper_2505_00232_b200 as P
    return P


def spec(N, K, bits, group):
    return C.LayerSpec("t", N, K, bits, group, *((-8, 7) if bits == 4 else (-128, 127)))


def route(P, Ns, K, bits, group, M, gated):
    ds = (type(P.Desc(8, 32, 8, 0).c()) * len(Ns))(*[P.Desc(N, K, bits, group).c() for N in Ns])
    out = (ctypes.c_int32 * 5)()
    assert P.lib.qlinear_debug_route(ds, len(Ns), M, gated, SMS, out, 5) >= 3
    return list(out)


def test_the_calls_below_get_these_plans(P):
    assert [route(P, [N], K, b, g, M, 0)[:3] for M, N, K, b, g, _, _ in PLAIN] == [[PAIR_TA, w, p] for *_, w, p in PLAIN]
    assert [route(P, [N, N], K, b, g, M, 1)[:3] for M, N, K, b, g, _ in GATED] == [[PAIR_TA, w, 1] for *_, w in GATED]
    assert [route(P, [N, N], K, b, g, M, 1)[:3] for M, N, K, b, g, *_ in TWO_ACCUMULATORS] == [[PAIR_TA, w, 1] for *_, w, _ in TWO_ACCUMULATORS]
    rounds = {-(-(-(-N // 256) * -(-M // w)) // (SMS // 2)) for M, N, *_, w, _ in TWO_ACCUMULATORS}
    assert rounds == {1, 2} and all(-(-N // 256) * -(-M // 256) < SMS // 2 for M, N, *_ in TWO_ACCUMULATORS)


def test_calls_with_int8_activations_get_these_plans(P):
    out = (ctypes.c_int32 * 4)()

    def plan(M, N, K, bits, group=0):
        n = P.lib.qlinear_debug_plan_a8(ctypes.byref(P.Desc(N, K, bits, group).c()), M, SMS, out, 4)
        return list(out)[:n]
    assert [plan(*c) for c, _ in A8_PARTS] == [[PAIR_TA, *p] for _, p in A8_PARTS]
    assert [plan(*c)[:3] for c, _ in A8_DECODE] == [[1, *p] for _, p in A8_DECODE]
    # refused: 9 to 128 tokens, K no multiple of 128, an odd number of row super-blocks, groups, rows that the scratch does not hold
    assert [plan(*c) for c in ((100, 256, 256, 8), (300, 256, 160, 8), (300, 128, 256, 8), (300, 256, 256, 4, 32), (5000, 256, 16384, 8))] == [[]] * 5


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K,bits,group", [c[:5] for c in PLAIN])
def test_plain(P, M, N, K, bits, group):
    import torch
    q, s = C.layer_weights(8100 + M, spec(N, K, bits, group))
    x = C.layer_activations(8100 + M, spec(N, K, bits, group), M)
    lin = P.QLinear.from_weights(q, s, bits, group, device="cuda:0")
    xd = torch.from_numpy(x).cuda()
    guard = torch.full((M + 2, N), -7.0, dtype=torch.float16, device="cuda")
    y = lin.forward(xd, out=guard[1:-1])
    assert torch.equal(y, lin.forward(xd)) and (guard[0] == -7.0).all() and (guard[-1] == -7.0).all()
    assert lin.device_status() == (0, 0)
    y64, A, _ = O.linear(x, q, s, group)
    d = np.abs(y.cpu().numpy().astype(np.float64) - y64)
    assert (d <= O.ELEM_TOL * A).all() and np.linalg.norm(d) <= O.REL_L2_TOL * np.linalg.norm(y64)


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K,bits,group", [c[:5] for c in GATED] + GATED_ON_NARROW)
def test_gated(P, M, N, K, bits, group):
    import torch
    from tests.test_gated_gpu import assert_gated
    gw, uw = (C.layer_weights(8200 + M + i, spec(N, K, bits, group)) for i in range(2))
    x = C.layer_activations(8200 + M, spec(N, K, bits, group), M)
    lg, lu = (P.QLinear.from_weights(q, s, bits, group, device="cuda:0") for q, s in (gw, uw))
    xd = torch.from_numpy(x).cuda()
    y = P.qlinear_forward_gated(lg, lu, xd, "silu")
    assert torch.equal(y, P.qlinear_forward_gated(lg, lu, xd, "silu")) and lg.device_status() == (0, 0)
    rows = np.r_[0:300, N - 300:N]
    assert_gated(y.cpu().numpy()[:, rows], x, (gw[0][rows], gw[1][rows]), (uw[0][rows], uw[1][rows]), group, "silu")


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K,bits,group,width,act", TWO_ACCUMULATORS)
def test_two_accumulators(P, M, N, K, bits, group, width, act):
    import torch
    from tests.test_gated_gpu import assert_gated
    gw, uw = (C.layer_weights(8400 + M + i, spec(N, K, bits, group)) for i in range(2))
    x = C.layer_activations(8400 + M, spec(N, K, bits, group), M)
    lg, lu = (P.QLinear.from_weights(q, s, bits, group, device="cuda:0") for q, s in (gw, uw))
    xd = torch.from_numpy(x).cuda()
    guard = torch.full((M + 2, N), -7.0, dtype=torch.float16, device="cuda")
    y = P.qlinear_forward_gated(lg, lu, xd, act, out=guard[1:-1])
    again = [P.qlinear_forward_gated(lg, lu, xd, act) for _ in range(20)]
    assert all(torch.equal(y, a) for a in again) and lg.device_status() == (0, 0) and (guard[0] == -7.0).all() and (guard[-1] == -7.0).all()
    rows = np.r_[0:300, N // 2:N // 2 + 100, N - 300:N] if N > 700 else np.r_[0:N]
    assert_gated(y.cpu().numpy()[:, rows], x, (gw[0][rows], gw[1][rows]), (uw[0][rows], uw[1][rows]), group, act)


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K,bits", A8 + [c for c, _ in A8_PARTS])
def test_integer_form(P, M, N, K, bits):
    import torch
    from tests.test_a8_gpu import assert_a8
    q, s = C.layer_weights(8300 + M, spec(N, K, bits, 0))
    x = C.layer_activations(8300 + M, spec(N, K, bits, 0), M)
    lin = P.QLinear.from_weights(q, s, bits, 0, device="cuda:0")
    xd = torch.from_numpy(x).cuda()
    y = lin.forward_a8(xd)
    again = [lin.forward_a8(xd) for _ in range(10)]
    assert all(torch.equal(y, a) for a in again) and lin.device_status() == (0, 0)
    rows = np.r_[0:128, N - 128:N] if N > 2304 else np.r_[0:N]
    assert_a8(y.cpu().numpy()[:, rows], x, q[rows], s[rows], 0)


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K,bits,group", [c for c, _ in A8_DECODE[6:]])
def test_integer_decode_in_clusters_of_each_size(P, M, N, K, bits, group):
    import torch
    from tests.test_a8_gpu import assert_a8
    q, s = C.layer_weights(8500 + M + N, spec(N, K, bits, group))
    x = C.layer_activations(8500 + M + N, spec(N, K, bits, group), M)
    lin = P.QLinear.from_weights(q, s, bits, group, device="cuda:0")
    xd = torch.from_numpy(x).cuda()
    y = lin.forward_a8(xd)
    assert all(torch.equal(y, lin.forward_a8(xd)) for _ in range(10))
    assert_a8(y.cpu().numpy(), x, q, s, group)
