"""The tile widths of the value product of many rows (16, 24, 32 and 64 rows to a tile, the last two shared by two groups of warps), with
remainders in rows, positions and channels, against the CPU oracle on a B200."""
import numpy as np
import pytest

from oracle import qlinear_oracle as O
from workloads import generators as gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_h,cache,R", [(64, 96, 17), (128, 1056, 50), (256, 2080, 129), (128, 4096, 250), (96, 1312, 460), (160, 704, 1100), (128, 1024, 2050), (256, 2080, 2047)])
def test_value_product_tiles(_built_library, d_h, cache, R):
    import torch
    import paper_2505_00232_b200 as P
    T = cache - 5
    kv = P.KVCache(cache, d_h, "cuda:0")
    v = gen.normal_fp16(6100 + R, 1, (T, d_h))
    kv.append(torch.from_numpy(v).cuda(), torch.from_numpy(v).cuda())
    prob = (gen.normal_fp16(6100 + R, 2, (R, cache)).astype(np.float32) ** 2 / 64).astype(np.float16)
    prob[:, T:] = 0
    guard = torch.full((R + 2, d_h), -7.0, dtype=torch.float16, device="cuda")
    p, tmp = torch.from_numpy(prob).cuda(), torch.empty((R, cache), dtype=torch.float16, device="cuda")
    P.binding._check(P.lib.qlinear_kv_output(kv.v._h, p.data_ptr(), kv.v_scale.data_ptr(), tmp.data_ptr(), guard[1:].data_ptr(), R, torch.cuda.current_stream().cuda_stream), "qlinear_kv_output")
    out = kv.output(p)
    assert torch.equal(out, guard[1:-1]) and (guard[0] == -7.0).all() and (guard[-1] == -7.0).all()
    v_q, v_s = O.kv_quantize_rows(v)
    folded = (prob[:, :T].astype(np.float32) * v_s.reshape(-1).astype(np.float32)).astype(np.float16)   # one fp16 rounding, as the kernel makes it
    y64, A, _ = O.kv_output(folded, np.ascontiguousarray(v_q.T), np.ones(d_h, np.float16))
    ok, rel, worst = O.check_against(out.cpu().numpy(), y64, A)
    assert ok, (rel, worst)
