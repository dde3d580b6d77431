"""Gated pairs of more than 128 tokens: the estimates that choose between the kernels, against times measured on a B200 (consecutive launches,
weights out of HBM), evaluated without a device."""
import ctypes

import pytest

SMS = 148
NARROW, PAIR_TA, PAIR = 5, 6, 7
# ((channels, K, bits, group, tokens), the kernel that serves the call, us it took)
ONE_ACCUMULATOR = [((12800, 128, 4, 32, 1410), PAIR_TA, 39.70), ((7936, 128, 4, 0, 1032), PAIR_TA, 23.56), ((11744, 128, 8, 0, 1373), PAIR_TA, 34.91),
                   ((14336, 4096, 4, 32, 777), PAIR_TA, 162.1), ((9216, 2304, 4, 32, 777), PAIR_TA, 57.77)]


# (beside each: us on the kernel that the estimates must not choose)
TWO_ACCUMULATORS = [((9440, 1536, 8, 0, 131), NARROW, 16.74),             # 20.5
                    ((7424, 1152, 8, 0, 176), NARROW, 14.78),             # 16.7
                    ((6144, 1120, 8, 0, 330), NARROW, 16.11),             # 18.1
                    ((9216, 1120, 8, 0, 130), NARROW, 14.06),             # 17.2
                    ((3464, 6336, 4, 32, 322), NARROW, 54.15),            # 60.2
                    ((6400, 7168, 8, 0, 426), NARROW, 97.06),             # 125.1
                    ((4096, 128, 4, 32, 873), PAIR_TA, 10.42),            # 13.2
                    ((4096, 128, 8, 0, 920), PAIR_TA, 11.12),             # 13.7 (two rounds)
                    ((9216, 2304, 4, 32, 300), PAIR_TA, 28.7),            # 43.6
                    ((1792, 1984, 4, 32, 1518), PAIR_TA, 25.95),          # 39.1
                    ((3040, 2624, 8, 0, 848), PAIR_TA, 30.68),            # 54.5
                    ((768, 4608, 8, 0, 3800), PAIR_TA, 47.31),            # 79.7
                    ((1000, 512, 8, 0, 257), NARROW, 7.73), ((3072, 4096, 4, 32, 1500), PAIR, 69.3)]   # 8.7, 81.9


@pytest.fixture(scope="module")
def route(_built_library):
    import paper_2505_00232_b200 as P

    def call(N, K, bits, group, M):
        ds = (type(P.Desc(8, 32, 8, 0).c()) * 2)(*[P.Desc(N, K, bits, group).c()] * 2)
        out = (ctypes.c_int32 * 5)()
        assert P.lib.qlinear_debug_route(ds, 2, M, 1, SMS, out, 5) == 5
        return list(out)
    return call


@pytest.mark.parametrize("shape,kernel,us", ONE_ACCUMULATOR + TWO_ACCUMULATORS)
def test_the_estimate_is_of_the_launch_that_runs(route, shape, kernel, us):
    """Within the spread of the fit (0.92 to 1.20)."""
    r = route(*shape)
    assert r[0] == kernel and 0.9 <= us / (r[3 if kernel == NARROW else 4] / 1000) <= 1.2, r
