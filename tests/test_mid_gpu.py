"""The kernel for a batch of tokens (9 to 64) and for the value product of many query rows, against the CPU oracle, on a
B200: edges of its token blocks, of the 128-channel super-blocks and of its two-chunk stages, with and without a K split."""
import numpy as np
import pytest

from oracle import qlinear_oracle as O
from workloads import configs as C
from workloads import generators as gen

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


@pytest.mark.parametrize("bits,group", [(4, 32), (4, 0), (4, 128), (8, 0)])
@pytest.mark.parametrize("M", [9, 16, 17, 24, 25, 32, 33, 48, 64])
@pytest.mark.parametrize("N,K", [(8, 128), (136, 384), (264, 2048), (640, 1152)])
def test_layer_group_and_gated_match_the_oracle(P, torch, M, N, K, bits, group):
    """One layer, three layers in one launch (of different widths), and the gated pair; K not a whole number of stages
    (1152 = 9 x 128 is odd in chunks of 64 for int4), a last super-block with 8 channels."""
    if not group:
        K -= 32 if N != 8 else 96                                        # a last chunk (int4) or stage (int8) that is half padding
    specs = [spec(n, K, bits, group) for n in (N, N, N + 128)]
    w = [C.layer_weights(6100 + M + N + K + i, s) for i, s in enumerate(specs)]
    x = C.layer_activations(6100 + M, specs[0], M)
    lins = [P.QLinear.from_weights(q, s, bits, group, device="cuda:0") for q, s in w]
    xd = torch.from_numpy(x).cuda()
    one = lins[0].forward(xd)
    many = P.qlinear_forward_group(lins, xd)
    gated = P.qlinear_forward_gated(lins[0], lins[1], xd, "silu")
    torch.cuda.synchronize()
    assert lins[0].device_status() == (0, 0)
    for y, (q, s) in zip(many, w):
        y64, A, _ = O.linear(x, q, s, group)
        ok, rel, worst = O.check_against(y.cpu().numpy(), y64, A)
        assert ok, (rel, worst)
    y64, A, _ = O.linear(x, *w[0], group)                                # (its own K split: another order of sums than in the group)
    ok, rel, worst = O.check_against(one.cpu().numpy(), y64, A)
    assert ok, (rel, worst)
    g64, bound, _ = O.gated_linear(x, *w[0], *w[1], group, "silu")
    ok, rel, worst = O.check_gated(gated.cpu().numpy(), g64, bound)
    assert ok, (rel, worst)
    assert torch.equal(one, lins[0].forward(xd)) and torch.equal(gated, P.qlinear_forward_gated(lins[0], lins[1], xd, "silu"))


def test_nothing_is_written_outside_the_output(P, torch):
    layer = spec(264, 256, 4, 32)
    q, s = C.layer_weights(6300, layer)
    lin = P.QLinear.from_weights(q, s, 4, 32, device="cuda:0")
    M = 19
    buf = torch.full((M + 2, 264), 7.0, dtype=torch.float16, device="cuda")
    lin.forward(torch.from_numpy(C.layer_activations(6300, layer, M)).cuda(), out=buf[1:M + 1])
    torch.cuda.synchronize()
    assert (buf[0] == 7).all() and (buf[M + 1] == 7).all() and not (buf[1:M + 1] == 7).all()


@pytest.mark.parametrize("d_h,cache,T,R", [(64, 96, 96, 9), (128, 1280, 1031, 17), (256, 512, 300, 24), (128, 2080, 2080, 33), (128, 4096, 3256, 1024)])
def test_value_product_of_many_rows(P, torch, d_h, cache, T, R):
    """out = P V with the per-token value scales folded into the probabilities inside the kernel, one fp16 rounding each."""
    v = (gen.normal_fp16(6400 + T, 2, (T, d_h)) * gen.normal_fp16(6400 + T, 4, (T, 1))).astype(np.float16)
    v[5] = 0
    kv = P.KVCache(cache, d_h)
    vd = torch.from_numpy(v).cuda()
    kv.append(vd, vd)
    p = np.exp(2 * gen.normal_fp16(6400 + R, 3, (R, T)).astype(np.float64))
    prob = np.zeros((R, cache), np.float16)
    prob[:, :T] = p / p.sum(axis=1, keepdims=True)
    out = kv.output(torch.from_numpy(prob).cuda())
    torch.cuda.synchronize()
    assert kv.v.device_status() == (0, 0)
    v_q, v_s = O.kv_quantize_rows(v)
    folded = (prob[:, :T].astype(np.float32) * v_s.astype(np.float32)).astype(np.float16)
    y64, A, _ = O.kv_output(folded, np.ascontiguousarray(v_q.T), np.ones(d_h, np.float16))
    ok, rel, worst = O.check_against(out.cpu().numpy(), y64, A)
    assert ok, (rel, worst)


def test_value_product_keeps_the_limit_on_its_output(P, torch):
    """2^31 output elements: refused like a forward call of that size (the buffers have the full size all the same)."""
    kv = P.KVCache(32, 65536)
    R = 32768
    prob = torch.zeros((R, 32), dtype=torch.float16, device="cuda")
    with pytest.raises(P.QLinearError) as err:
        kv.output(prob)
    assert err.value.status == P.QL_ERR_INVALID_ARG
    assert kv.output(prob[:100]).shape == (100, 65536)


@pytest.mark.parametrize("d_h,cache,R,large", [(512, 2048, 4096, False), (512, 4096, 4096, True), (1024, 256, 4096, True), (1024, 1024, 2048, False), (1024, 4096, 1024, True), (640, 4096, 4096, False)])
def test_value_product_on_both_sides_of_the_prefill_kernel(P, torch, d_h, cache, R, large):
    """Wide heads and many rows: the scales as a pass of their own (into the scratch argument) and the prefill kernel, where that is
    faster; 640 channels are an odd number of super-blocks.  Both routes against the oracle, on some of the rows."""
    import ctypes
    kv = P.KVCache(cache, d_h)
    v = (gen.normal_fp16(6500 + cache, 2, (cache, d_h)) * gen.normal_fp16(6500 + cache, 4, (cache, 1))).astype(np.float16)
    vd = torch.from_numpy(v).cuda()
    kv.append(vd, vd)
    prob = (torch.rand((R, cache), device="cuda") / cache).half()
    tmp = torch.full((R, cache), 7.0, dtype=torch.float16, device="cuda")
    out = torch.empty((R, d_h), dtype=torch.float16, device="cuda")
    vp = ctypes.c_void_p
    assert P.lib.qlinear_kv_output(kv.v._h, vp(prob.data_ptr()), vp(kv.v_scale.data_ptr()), vp(tmp.data_ptr()), vp(out.data_ptr()), R, vp(torch.cuda.current_stream().cuda_stream)) == 0
    torch.cuda.synchronize()
    assert kv.v.device_status() == (0, 0)
    assert bool((tmp == 7).all()) != large
    rows = [0, 1, 63, 64, 255, 256, R - 1]
    v_q, v_s = O.kv_quantize_rows(v)
    folded = (prob[rows].cpu().numpy().astype(np.float32) * v_s.astype(np.float32)).astype(np.float16)
    y64, A, _ = O.kv_output(folded, np.ascontiguousarray(v_q.T), np.ones(d_h, np.float16))
    ok, rel, worst = O.check_against(out[rows].cpu().numpy(), y64, A)
    assert ok, (rel, worst)


# (N, K, bits, group, M, whether the batch kernel takes it): both sides of each line of the rule
LINES = [(12000, 4096, 4, 32, 48, False), (11584, 4096, 4, 32, 48, True), (7424, 4096, 4, 32, 64, False), (7168, 4096, 4, 32, 64, True),
         (5888, 4096, 8, 0, 49, False), (5632, 4096, 8, 0, 49, True), (14336, 4096, 4, 0, 32, True), (2304, 2304, 8, 0, 65, False)]


@pytest.mark.parametrize("N,K,bits,group,M,mid", LINES)
def test_lines_between_the_batch_kernel_and_the_prefill_kernel(P, torch, N, K, bits, group, M, mid):
    """The shape picks the kernel that was measured to be faster; both give the layer."""
    import ctypes
    layer = spec(N, K, bits, group)
    q, s = C.layer_weights(6600 + N, layer)
    x = C.layer_activations(6600 + M, layer, M)
    lin = P.QLinear.from_weights(q, s, bits, group, device="cuda:0")
    assert P.lib.qlinear_debug_takes_batch_kernel((ctypes.c_void_p * 1)(lin._h), 1, M) == mid
    y = lin.forward(torch.from_numpy(x).cuda())
    torch.cuda.synchronize()
    assert lin.device_status() == (0, 0)
    rows = np.r_[0:64, N - 64:N]
    y64, A, _ = O.linear(x, q[rows], s[rows], group)
    ok, rel, worst = O.check_against(y.cpu().numpy()[:, rows], y64, A)
    assert ok, (rel, worst)


def test_gated_pair_between_the_lines_needs_no_scratch(P, torch):
    """64 tokens, 38 million weights: a forward call of that size is the prefill kernel's, the gated pair stays one launch of the
    batch kernel: gated calls on two streams that are not ordered against each other, which may not share the device scratch."""
    layer = spec(8192, 2304, 4, 32)
    w = [C.layer_weights(6700 + i, layer) for i in range(2)]
    gate, up = (P.QLinear.from_weights(q, s, 4, 32, device="cuda:0") for q, s in w)
    xs = [torch.from_numpy(C.layer_activations(6700 + i, layer, 64)).cuda() for i in range(2)]
    first = [P.qlinear_forward_gated(gate, up, x, "silu") for x in xs]
    streams = [torch.cuda.Stream() for _ in range(2)]
    outs = [torch.empty_like(f) for f in first]
    torch.cuda.synchronize()
    for _ in range(50):
        for x, o, st in zip(xs, outs, streams):
            P.qlinear_forward_gated(gate, up, x, "silu", out=o, stream=st)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(first, outs)) and gate.device_status() == (0, 0)
    rows = np.r_[0:64, 8128:8192]
    g64, bound, _ = O.gated_linear(xs[0].cpu().numpy(), w[0][0][rows], w[0][1][rows], w[1][0][rows], w[1][1][rows], 32, "silu")
    ok, rel, worst = O.check_gated(first[0].cpu().numpy()[:, rows], g64, bound)
    assert ok, (rel, worst)
