"""The tensor-core kernel of the score product of many rows, against the CPU oracle, on a B200: a last token block and a last super-block
that are not full, CTAs whose tiles span heads and super-blocks, each head dimension."""
import numpy as np
import pytest

from oracle import qlinear_oracle as O

pytestmark = pytest.mark.gpu


CASES = [(2, 64, 8160, 8000, 1000), (3, 128, 4064, 3000, 1001), (9, 128, 2080, 2080, 2017), (2, 256, 992, 900, 4000), (1, 128, 160, 160, 20001)]


@pytest.mark.parametrize("n_heads,d_h,cache,T,R", CASES)
def test_scores_of_very_many_rows(_built_library, n_heads, d_h, cache, T, R):
    import torch
    import paper_2505_00232_b200 as P
    rng = np.random.default_rng(cache + R)
    k = (rng.standard_normal((n_heads, T, d_h)) * rng.uniform(0.2, 3.0, size=(n_heads, T, 1))).astype(np.float16)
    q = rng.standard_normal((n_heads, R, d_h)).astype(np.float16)
    heads = P.KVHeads(n_heads, cache, d_h)
    heads.append(torch.from_numpy(k).cuda(), torch.from_numpy(k).cuda())
    buf = torch.full((n_heads * R + 2, cache), 7.0, dtype=torch.float16, device="cuda")
    sc = buf[1:-1].view(n_heads, R, cache)
    heads.scores_raw(torch.from_numpy(q).cuda().data_ptr(), sc.data_ptr(), R)
    torch.cuda.synchronize()
    assert heads.heads[0].k.device_status() == (0, 0)
    assert (buf[0] == 7).all() and (buf[-1] == 7).all() and (sc[:, :, T:] == 0).all()
    rows = np.unique(np.r_[0:70, R // 2:R // 2 + 64, R - 70:R])
    for h in range(n_heads):
        k_q, k_s = O.kv_quantize_rows(k[h])
        y64, A, _ = O.linear(q[h][rows], k_q, k_s.reshape(-1, 1), 0)
        ok, rel, worst = O.check_against(sc[h, :, :T].cpu().numpy()[rows], y64, A)
        assert ok, (h, rel, worst)
