"""Readers of a KV cache that run ahead of the append before them: only the tokens of that append are held back, so its first and last
token are put on the edges of what the readers hold back (super-blocks of 128 tokens, chunks of 32), on a B200."""
import numpy as np
import pytest

from oracle import qlinear_oracle as O

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


@pytest.mark.parametrize("n_heads,d_h,cache", [(8, 128, 1280), (2, 64, 4096), (3, 256, 2080)])
@pytest.mark.parametrize("pos,n_new", [(0, 1), (31, 1), (32, 1), (127, 1), (127, 2), (128, 1), (640, 128), (700, 97), (1279, 1)])
def test_products_of_tokens_appended_just_before(P, torch, n_heads, d_h, cache, pos, n_new):
    """append to one cache, then to another, then the products of the first: captured as a graph and replayed on new tokens, against the
    same calls with the host waiting in between; the last state against the oracle."""
    T = min(cache, 1280)
    rng = np.random.default_rng(pos + d_h)
    start = torch.from_numpy((rng.standard_normal((n_heads, T, d_h))).astype(np.float16)).cuda()
    pair = [[P.KVHeads(n_heads, cache, d_h) for _ in range(2)] for _ in range(2)]
    for caches in pair:
        for kv in caches:
            kv.append(start, start)
    q = torch.from_numpy(rng.standard_normal((n_heads, 4, d_h)).astype(np.float16)).cuda()
    prob = torch.full((n_heads, 4, cache), 2.0 ** -10, dtype=torch.float16, device="cuda")
    kn, vn = (torch.zeros((n_heads, n_new, d_h), dtype=torch.float16, device="cuda") for _ in range(2))

    def step(caches, wait):
        out = []
        for kv in caches:
            kv.length = pos
            kv.append(kn, vn)
            wait()
        for kv in caches:
            out += [kv.output(prob), kv.scores(q)]
            wait()
        return out
    step(pair[0], lambda: None)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = step(pair[0], lambda: None)
    for _ in range(8):
        kn.copy_(torch.randn_like(kn) * 3)
        vn.copy_(torch.randn_like(vn) * 3)
        graph.replay()
        torch.cuda.synchronize()
        want = step(pair[1], torch.cuda.synchronize)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(got, want))
    for h in (0, n_heads - 1):
        k = start[h].cpu().numpy().copy()
        k[pos:pos + n_new] = kn[h].cpu().numpy()
        k_q, k_s = O.kv_quantize_rows(k)
        y64, A, _ = O.linear(q[h].cpu().numpy(), k_q, k_s.reshape(-1, 1), 0)
        ok, rel, worst = O.check_against(got[1][h, :, :T].cpu().numpy(), y64, A)
        assert ok, (h, rel, worst)


BATCH = [(4, 96, 16384, 64), (2, 96, 15680, 49), (1, 96, 41728, 33), (2, 32, 46880, 64), (2, 160, 16384, 64)]


@pytest.mark.parametrize("n_heads,d_h,cache,R", BATCH)
def test_scores_of_a_batch_of_rows_see_the_scales_appended_just_before(P, torch, n_heads, d_h, cache, R):
    """Head dimensions that the row kernels do not take and many positions: the batch kernels.  On the one with the weights in tensor
    memory (test_routes_gpu.py has it serve them) these are launches of one K part, and (up to 128 of K) of a step for one of its two groups of
    warps only: the other one waits for nothing before its outputs.  Append and scores captured and replayed on new tokens, against the same calls with the host waiting in between."""
    T, n_new = cache - 100, 64
    start = torch.randn((n_heads, T, d_h), device="cuda").half()
    pair = [P.KVHeads(n_heads, cache, d_h) for _ in range(2)]
    for kv in pair:
        kv.append(start, start)
    q = torch.randn((n_heads, R, d_h), device="cuda").half()
    kn = torch.zeros((n_heads, n_new, d_h), dtype=torch.float16, device="cuda")

    def step(kv, wait):
        kv.length = T
        kv.append(kn, kn)
        wait()
        return kv.scores(q)
    step(pair[0], lambda: None)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = step(pair[0], lambda: None)
    for i in range(20):
        kn.copy_(torch.randn_like(kn) * (0.1 if i & 1 else 10.0))
        graph.replay()
        torch.cuda.synchronize()
        want = step(pair[1], torch.cuda.synchronize)
        torch.cuda.synchronize()
        assert torch.equal(got, want)
    assert pair[0].heads[0].k.device_status() == (0, 0)
    k_q, k_s = O.kv_quantize_rows(kn[0].cpu().numpy())
    y64, A, _ = O.linear(q[0].cpu().numpy(), k_q, k_s.reshape(-1, 1), 0)
    ok, rel, worst = O.check_against(got[0, :, T:T + n_new].cpu().numpy(), y64, A)
    assert ok, (rel, worst)


ALL = 0x7fffffe0                                        # what qlinear_debug_kv_hold gives as the end of "every token"


def hold(P, heads, stream):
    """The tokens that a decode reader of all heads' scores on this stream holds back."""
    import ctypes
    first, end = ctypes.c_int32(-1), ctypes.c_int32(-1)
    assert P.lib.qlinear_debug_kv_hold(heads._hk, heads.n, stream.cuda_stream, ctypes.byref(first), ctypes.byref(end)) == 0
    return first.value, end.value


def append_at(heads, pos, tokens, stream=None):
    heads.length = pos
    heads.append(tokens, tokens, stream=stream)


def test_readers_hold_back_whatever_may_be_in_flight(P, torch):
    """Only the tokens of the last append where that one was enqueued on the reader's stream and in its capture; everything elsewhere."""
    kv = P.KVHeads(2, 256, 64)
    new = torch.randn((2, 3, 64), device="cuda").half()
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    for s in (s1, s2):
        s.wait_stream(torch.cuda.current_stream())
    assert hold(P, kv, s1) == (0, 0)
    append_at(kv, 10, new, s1)
    assert hold(P, kv, s1) == (10, 13) and hold(P, kv, s2) == (0, ALL)
    append_at(kv, 13, new, s1)
    assert hold(P, kv, s1) == (13, 16)
    s2.wait_stream(s1)
    append_at(kv, 16, new, s2)                          # s1's own append is now one of those that may be in flight for a reader there
    assert hold(P, kv, s1) == (0, ALL) and hold(P, kv, s2) == (16, 19)
    append_at(kv, 20, new, torch.cuda.default_stream())
    assert hold(P, kv, torch.cuda.default_stream()) == (20, 23) and hold(P, kv, s1) == (0, ALL)

    class PerThread:
        cuda_stream = 2                                 # cudaStreamPerThread: another stream in every thread
    assert hold(P, kv, PerThread) == (0, ALL)
    torch.cuda.synchronize()
    append_at(kv, 30, new, s1)
    with torch.cuda.graph(torch.cuda.CUDAGraph(), stream=s1):
        assert hold(P, kv, s1) == (0, ALL)              # a reader without an append of its own capture
        append_at(kv, 40, new, s1)
        assert hold(P, kv, s1) == (40, 43)
        side = torch.cuda.Stream()
        side.wait_stream(s1)
        append_at(kv, 50, new, side)
        append_at(kv, 53, new, s1)
        assert hold(P, kv, s1) == (0, ALL) and hold(P, kv, side) == (0, ALL)
        s1.wait_stream(side)
        append_at(kv, 56, new, s1)
        assert hold(P, kv, s1) == (0, ALL)              # (for good, in this capture)
    assert hold(P, kv, s1) == (0, ALL)                  # the capture's last append has not run: the one in flight is another
    append_at(kv, 60, new, s1)
    assert hold(P, kv, s1) == (60, 63)
    torch.cuda.synchronize()


def test_an_append_that_is_not_launched_leaves_the_last_one(P, torch):
    """A launch into an invalidated capture fails on the host; what may be in flight is still the append before it."""
    import ctypes
    cu = ctypes.CDLL("libcuda.so.1")
    kv = P.KVHeads(1, 128, 64)
    new = torch.randn((1, 2, 64), device="cuda").half()
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    append_at(kv, 5, new, s)
    torch.cuda.synchronize()
    st, graph = ctypes.c_void_p(s.cuda_stream), ctypes.c_void_p()
    assert cu.cuStreamBeginCapture_v2(st, 2) == 0
    assert cu.cuStreamSynchronize(st) != 0              # not allowed while capturing: invalidates the capture
    with pytest.raises(P.QLinearError) as err:
        append_at(kv, 9, new, s)
    assert err.value.status == P.QL_ERR_CUDA
    assert cu.cuStreamEndCapture(st, ctypes.byref(graph)) != 0
    assert hold(P, kv, s) == (5, 7)
    append_at(kv, 9, new, s)
    assert hold(P, kv, s) == (9, 11)
    torch.cuda.synchronize()


@pytest.mark.parametrize("d_h", [64, 128, 256])
@pytest.mark.parametrize("case", ["capture_between", "two_streams", "two_branches"])
def test_a_reader_behind_an_append_that_is_not_the_last_recorded(P, torch, case, d_h):
    """The append that a reader follows in its stream is still waiting (for a kernel that takes milliseconds) when another one has been
    recorded: in a capture that has not run, or on a second stream.  Scores and values against the same calls with the host waiting."""
    H, cache, T = 4, 2048, 1024
    start = torch.randn((H, T, d_h), device="cuda").half()
    q = torch.randn((H, 4, d_h), device="cuda").half()
    prob = torch.full((H, 4, cache), 2.0 ** -10, dtype=torch.float16, device="cuda")
    a = torch.zeros((H, 700, d_h), dtype=torch.float16, device="cuda")
    b = torch.zeros((H, 1, d_h), dtype=torch.float16, device="cuda")
    kv, ref = (P.KVHeads(H, cache, d_h) for _ in range(2))
    for c in (kv, ref):
        append_at(c, 0, start)
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()

    def read(c):
        with torch.cuda.stream(s1):
            return [c.scores(q, stream=s1), c.output(prob, stream=s1)]

    def branches():
        """(captured on s1) a on s1 and b on a branch, joined, read."""
        s2.wait_stream(s1)
        append_at(kv, 100, a, s1)
        append_at(kv, 900, b, s2)
        s1.wait_stream(s2)
        return read(kv)
    append_at(kv, 900, b, s1)
    read(kv)                                            # (first launches happen outside the capture)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    if case == "two_branches":
        with torch.cuda.graph(graph, stream=s1):
            got = branches()
    for _ in range(4):
        a.copy_(torch.randn_like(a) * 3)
        b.copy_(torch.randn_like(b) * 3)
        for c in (kv, ref):
            append_at(c, 0, start)
        torch.cuda.synchronize()
        if case == "two_branches":
            graph.replay()
        else:
            with torch.cuda.stream(s1):
                torch.cuda._sleep(10_000_000)
            append_at(kv, 100, a, s1)
            if case == "capture_between":
                with torch.cuda.stream(s2):
                    other = torch.cuda.CUDAGraph()
                    other.capture_begin(capture_error_mode="thread_local")
                    append_at(kv, 900, b, s2)
                    other.capture_end()
            else:
                append_at(kv, 900, b, s2)
                s1.wait_stream(s2)
            got = read(kv)
        torch.cuda.synchronize()
        append_at(ref, 100, a)
        if case != "capture_between":
            append_at(ref, 900, b)
        torch.cuda.synchronize()
        want = read(ref)
        torch.cuda.synchronize()
        assert all(torch.equal(x, y) for x, y in zip(got, want))
    assert kv.heads[0].k.device_status() == (0, 0)


# heads, d_h, new tokens: both sides of the line between two and four dimensions per lane, d_h not a multiple of a warp's slice
@pytest.mark.parametrize("n_heads,d_h,n_new", [(1, 32, 3), (3, 96, 40), (16, 128, 300), (8, 160, 40), (8, 160, 660), (2, 256, 5), (16, 256, 130), (2, 992, 3), (2, 992, 70), (1, 1024, 127), (4, 1024, 33)])
def test_appended_integers_and_scales_of_any_width(P, torch, n_heads, d_h, n_new):
    cache, pos = (n_new + 31) // 32 * 32 + 64, 37
    rng = np.random.default_rng(d_h + n_new)
    k, v = ((rng.standard_normal((n_heads, n_new, d_h)) * rng.uniform(0.1, 9.0, size=(n_heads, n_new, 1))).astype(np.float16) for _ in range(2))
    v[0, 1], k[n_heads - 1, 2] = 0, 2.0 ** -20                # a zero vector; a scale below fp16's range
    kv = P.KVHeads(n_heads, cache, d_h)
    kv.length = pos
    kv.append(torch.from_numpy(k).cuda(), torch.from_numpy(v).cuda())
    torch.cuda.synchronize()
    where = slice(pos, pos + n_new)
    for h, c in enumerate(kv.heads):
        k_q, k_s = O.kv_quantize_rows(k[h])
        v_q, v_s = O.kv_quantize_rows(v[h])
        got_k, got_v = c.k.debug_unpack().cpu().numpy(), c.v.debug_unpack().cpu().numpy()
        assert (got_k[where] == k_q).all() and (got_v[:, where] == v_q.T).all()
        assert (np.delete(got_k, np.r_[where], 0) == 0).all() and (np.delete(got_v, np.r_[where], 1) == 0).all()
        _, ks = P.qlinear_unpack(c.k.desc, c.k.packed.cpu().numpy())
        assert (ks.reshape(-1)[where].view(np.uint16) == k_s.view(np.uint16)).all()
        assert (c.v_scale.cpu().numpy()[where].view(np.uint16) == v_s.view(np.uint16)).all()
