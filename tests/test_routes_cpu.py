"""Which kernel serves which call: the dispatch evaluated without a device (qlinear_debug_route), for the cases of the GPU tests, so that a
change of a line between two kernels cannot silently empty a test.  The switches are read once per process: one child per setting."""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SMS = 148                                               # of a B200
DECODE, ROWS, ROWS_TC, MID, NARROW, PAIR_TA, PAIR, SINGLE, SEPARATE = range(1, 10)

CHILD = """
import ctypes, json, sys
sys.path.insert(0, {root!r})
import paper_2505_00232_b200 as P
from tests import test_gated_gpu, test_kv_append_gpu, test_mid_gpu, test_narrow_gpu, test_prefill_gpu, test_prefill_ta_gpu, test_scores_gpu

def route(Ns, K, bits, group, M, gated=0):
    ds = (type(P.Desc(8, 32, 8, 0).c()) * len(Ns))(*[P.Desc(N, K, bits, group).c() for N in Ns])
    out = (ctypes.c_int32 * 5)()
    assert P.lib.qlinear_debug_route(ds, len(Ns), M, gated, {sms}, out, 5) >= 1
    return list(out)

plain = lambda cases: [route([N], K, b, g, M) for M, N, K, b, g in cases]
pairs = lambda cases: [route([N, N], K, b, g, M, 1) for M, N, K, b, g in cases]
print(json.dumps({{
    "small": plain(test_prefill_gpu.SMALL), "tiles": plain(test_prefill_gpu.NARROW), "tiles_gated": pairs(test_prefill_gpu.NARROW_GATED),
    "groups": [route(Ns, K, b, g, M) for M, K, b, g, Ns in test_prefill_gpu.GROUPS],
    "ta": plain(test_prefill_ta_gpu.CASES), "widths": plain(test_prefill_ta_gpu.WIDTHS), "stress": plain(test_prefill_ta_gpu.STRESS),
    "fallback": route([2304, 2304], 2048, 4, 32, 96, 1), "fused": route([9728, 9728], 1024, 4, 32, 2048, 1),
    "gated": pairs([c[:5] for c in test_gated_gpu.CASES]),
    "late": [route([768], d, 8, 0, R) for d, R in ((96, 200), (512, 100), (512, 200), (384, 300))],
    "late_batch": [route([c], d, 8, 0, R) for _, d, c, R in test_kv_append_gpu.BATCH],
    "narrow_small": [[route([N], K, b, g, M), route([N, N + 136], K, b, g, M), route([N, N], K, b, g, M, 1)] for N, K, b, g, M in test_narrow_gpu.SMALL],
    "narrow_large": [route([N], K, b, g, M) for N, K, b, g, M in test_narrow_gpu.LARGE],
    "lines": [route([N], K, b, g, M) for N, K, b, g, M, _ in test_mid_gpu.LINES],
    "scores": [route([c], d, 8, 0, R) for _, d, c, _, R in test_scores_gpu.CASES]}}))
"""


def routes(**env):
    env = {**{k: v for k, v in os.environ.items() if not k.startswith("QLINEAR_")}, **env}
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT, sms=SMS)], check=True, env=env, cwd=ROOT, timeout=600, stdout=subprocess.PIPE)
    return json.loads(r.stdout)


@pytest.fixture(scope="module")
def by_rule(_built_library):
    return routes()


@pytest.fixture(scope="module")
def without_narrow(_built_library):
    return routes(QLINEAR_GEMM_NARROW="0")


@pytest.fixture(scope="module")
def always_narrow(_built_library):
    return routes(QLINEAR_GEMM_NARROW="2")


def kernels(rs):
    return [r[0] for r in rs]


def test_the_kernel_for_a_batch_serves_its_tests(by_rule, always_narrow):
    """Under the switch all of them, with both forms of the K split and every number of groups of warps; by the rule the large layers."""
    flat = [r for three in always_narrow["narrow_small"] for r in three] + always_narrow["narrow_large"]
    assert set(kernels(flat)) == {NARROW}
    assert {r[2] for r in flat} >= {1, 2, 4, 8} and min(r[1] for r in flat) == 16 and max(r[1] for r in flat) == 64
    assert kernels(by_rule["narrow_large"]) == [NARROW] * len(by_rule["narrow_large"])
    assert kernels(by_rule["late_batch"]) == [NARROW] * len(by_rule["late_batch"]) and {r[2] for r in by_rule["late_batch"]} == {1}


def test_the_score_kernel_of_many_rows_serves_its_tests(by_rule):
    assert kernels(by_rule["scores"]) == [ROWS_TC] * len(by_rule["scores"])


def test_the_prefill_kernels_serve_their_tests(without_narrow):
    """With the kernel for a batch of tokens switched off: both tile widths of the single-CTA kernel, the CTA-pair kernel whole and split
    into 2 and 4 K parts, both forms of the fused gating, the unfused one."""
    r = without_narrow
    big = [x for x in r["small"] if x[0] != MID]
    assert len(big) == 15 and {x[0] for x in big} == {SINGLE, PAIR_TA}
    assert {x[1] for x in big if x[0] == SINGLE} == {128, 256} and {x[2] for x in big if x[0] == PAIR_TA} >= {1, 2, 4}
    assert all(x[0] == PAIR_TA and x[2] > 1 for x in r["small"][-3:-1]) and r["small"][-1][:3] == [PAIR_TA, 256, 2]
    over = [x for c, x in zip(_widths(), r["widths"]) if c[0] > 64]
    assert set(kernels(over)) == {PAIR_TA} and {x[2] for x in over} == {1, 2, 4} and {x[1] for x in over} == {96, 128}
    assert kernels(r["ta"]) == [PAIR_TA] * len(r["ta"]) and kernels(r["stress"]) == [PAIR_TA] * len(r["stress"])
    assert [x[2] for x in r["stress"]] == [1, 1, 2, 1, 4]
    assert kernels(r["groups"]) == [PAIR_TA] * len(r["groups"])
    assert r["fallback"][0] == SEPARATE and r["fused"][0] == PAIR_TA
    assert kernels(r["gated"]) == [DECODE] * 5 + [PAIR] * 4 + [MID] + [SEPARATE] * 2
    assert kernels(r["late"]) == [PAIR_TA, PAIR_TA, PAIR_TA, PAIR_TA]


def test_the_batch_kernel_with_warp_level_mmas_serves_its_tests(by_rule, without_narrow):
    from tests import test_mid_gpu
    for c, x in zip(test_mid_gpu.LINES, without_narrow["lines"]):
        assert (x[0] == MID) == c[5], c
    assert {x[0] for c, x in zip(test_mid_gpu.LINES, by_rule["lines"]) if not c[5]} <= {NARROW, PAIR_TA}


def _widths():
    from tests import test_prefill_ta_gpu
    return test_prefill_ta_gpu.WIDTHS
