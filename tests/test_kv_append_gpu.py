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
