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

# (channels of the layers, K, bits, group, tokens, gated, kernel)
CLEAR = [([14336] * 2, 4096, 4, 32, 32, 1, NARROW), ([4096], 14336, 4, 32, 32, 0, NARROW), ([4096, 1024, 1024], 4096, 8, 0, 32, 0, NARROW),
         ([2304], 9216, 4, 32, 48, 0, NARROW), ([1024], 1024, 8, 0, 128, 0, NARROW), ([1024], 1024, 4, 32, 512, 0, NARROW),
         ([2688] * 2, 1024, 4, 32, 128, 1, NARROW), ([2680], 64, 4, 32, 411, 0, NARROW), ([512], 512, 4, 32, 16, 0, MID),
         ([1024], 1024, 8, 0, 24, 0, MID), ([9216] * 2, 2304, 4, 32, 16, 1, MID), ([11816] * 2, 64, 4, 0, 48, 1, MID), ([512] * 2, 2048, 4, 0, 32, 1, MID),
         ([4096], 14336, 4, 32, 2048, 0, PAIR_TA), ([14336] * 2, 4096, 4, 32, 777, 1, PAIR_TA), ([4096, 1024, 1024], 4096, 8, 0, 1024, 0, PAIR_TA),
         # what the smoke run has for the prefill kernels
         ([4096], 512, 4, 32, 1024, 0, PAIR_TA), ([128], 96, 8, 0, 300, 0, SINGLE), ([3072] * 2, 4096, 4, 32, 1500, 1, PAIR),
         ([6936], 10144, 4, 32, 1500, 0, SINGLE)]

# (d_h, cache, rows, kernel): both sides of the lines for scores of many rows
SCORE_LINES = [(64, 8192, 1024, ROWS_TC), (64, 8192, 896, ROWS), (128, 32768, 128, ROWS), (128, 32768, 129, ROWS_TC), (128, 8192, 512, ROWS_TC), (128, 8192, 448, ROWS),
               (256, 32768, 128, ROWS_TC), (256, 4096, 896, ROWS_TC), (256, 4096, 832, ROWS)]

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
    "clear": [route(*c[:6]) for c in {clear!r}],
    "score_lines": [route([c], d, 8, 0, R) for d, c, R, _ in {score_lines!r}],
    "lines": [route([N], K, b, g, M) for N, K, b, g, M, _ in test_mid_gpu.LINES],
    "scores": [route([c], d, 8, 0, R) for _, d, c, _, R in test_scores_gpu.CASES]}}))
"""


def routes(**env):
    env = {**{k: v for k, v in os.environ.items() if not k.startswith("QLINEAR_")}, **env}
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT, sms=SMS, clear=CLEAR, score_lines=SCORE_LINES)], check=True, env=env, cwd=ROOT, timeout=600, stdout=subprocess.PIPE)
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


def test_the_kernel_for_a_batch_serves_its_tests(always_narrow):
    """Under the switch all of them, with and without a K split, at the narrowest and the widest token block."""
    flat = [r for three in always_narrow["narrow_small"] for r in three] + always_narrow["narrow_large"]
    assert set(kernels(flat)) == {NARROW}
    assert {r[2] for r in flat} >= {1, 2, 4, 8} and min(r[1] for r in flat) == 16 and max(r[1] for r in flat) == 64
    assert kernels(always_narrow["late_batch"]) == [NARROW] * 5 and {r[2] for r in always_narrow["late_batch"]} == {1}


def test_calls_far_from_the_lines_go_to_the_faster_kernel(by_rule):
    """Both sides measured at twice the other's time or nearly so, except where the comment in gemm_route gives the figures."""
    assert kernels(by_rule["clear"]) == [c[-1] for c in CLEAR]


def test_the_score_kernel_of_many_rows_serves_its_tests(by_rule):
    assert kernels(by_rule["scores"]) == [ROWS_TC] * len(by_rule["scores"])
    assert kernels(by_rule["score_lines"]) == [c[-1] for c in SCORE_LINES]


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
