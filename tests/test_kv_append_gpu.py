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


@pytest.mark.parametrize("n_heads,d_h,cache,R", [(4, 96, 16384, 64), (2, 96, 15680, 49), (1, 96, 41728, 33), (2, 32, 46880, 64), (2, 160, 16384, 64)])
def test_scores_of_a_batch_of_rows_see_the_scales_appended_just_before(P, torch, n_heads, d_h, cache, R):
    """Head dimensions that the row kernels do not take, so many positions that the batch kernel with the weights in tensor memory serves the
    scores in one K part, and (up to 128 of K) a step for one of its two groups of warps only: the other one waits for nothing before
    its outputs.  Append and scores captured and replayed on new tokens, against the same calls with the host waiting in between."""
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
