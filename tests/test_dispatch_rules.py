"""Host rules that pick a kernel, over ranges of call sizes: the library is asked without a GPU."""
import ctypes

import pytest

from gpu_common import NARROW, UNITS, bwd_dq_grid, linear_schedule


@pytest.fixture(scope="module")
def lib():
    from paper_2609_35140_b200 import binding
    lib = binding.load()
    lib.tik_selftest_decode_cluster.argtypes = [ctypes.c_int64] + 4 * [ctypes.c_int]
    return lib


@pytest.mark.parametrize("sms", [148, 132])
def test_narrow_linear_is_one_wave_or_one_cta_per_row_tile(lib, sms):
    """A second wave of narrow CTAs repeats the whole chain over K: no shape gets one, except that row tiles beyond
    the number of SMs take a CTA each, which then holds all columns.  No CTA has more columns than there are."""
    taken = 0
    for T in list(range(1, 140)) + [255, 256, 257, 384, 640, 768, 1024, 2048, 2049, 3456, 5000, 8192, 18944, 20000, 100000]:
        for N in list(range(8, 1700, 8)) + list(range(4096, 9600, 64)):
            schedule, ctas, cols = linear_schedule(lib, T, 1536, N, sms)
            if schedule == NARROW:
                taken += 1
                tiles = -(-T // 128)
                assert ctas == -(-N // cols) * tiles and (ctas <= sms or ctas == tiles), (T, N, ctas, cols)
                assert cols < N + 16, (T, N, cols)
    assert taken > 10000

@pytest.mark.parametrize("N,cols", [(37888, 256), (37896, 128), (40960, 128), (55296, 128), (56832, 128), (56840, 256), (75776, 256)])
def test_wide_linear_of_65_to_128_rows_keeps_the_sms_at_work(lib, N, cols):
    """One pass over W: three rounds of 128 columns rather than two of 256 whose second is partly empty; 256 columns
    where their last round is as full."""
    for T in (65, 100, 128):
        assert linear_schedule(lib, T, 5120, N)[::2] == (UNITS, cols)


@pytest.mark.parametrize("max_clusters", [0, 1, 33, 37])
def test_clusters_only_while_all_of_them_run_at_once(lib, max_clusters):
    """A cluster decode whose clusters do not all fit takes a second wave: 1.5 to 2 times the time of the kernels
    without clusters.  How many fit is the device's answer (33 of four CTAs on 148 SMs), not SMs / 4."""
    for chunks in range(1, 60):
        got = lib.tik_selftest_decode_cluster(chunks, 4000, 8, 128, max_clusters)
        assert got == (4 if chunks <= max_clusters else 0), chunks
    for refused in ((4, 896, 8, 128), (4, 4000, 9, 128), (4, 4000, 8, 64)):
        assert lib.tik_selftest_decode_cluster(*refused, max_clusters) == 0


def test_dq_grid_order(lib):
    """Heads fastest only where that is no slower than one head after the other: K and V of all heads stay in L2, and few
    tiles of the grid are empty."""
    full = [(1, 8192, 32, 8, 128), (2, 4096, 32, 8, 128), (3, 1500, 8, 8, 128), (8, 4096, 12, 2, 128), (1, 16384, 28, 4, 128),
            (1, 10240, 16, 16, 128), (2, 4096, 32, 32, 128), (1, 20480, 8, 8, 128)]
    for S, L, Hq, Hkv, d in full:
        assert bwd_dq_grid(lib, S, S * L, L, Hq, Hkv, d)[0] is False, (S, L, Hq, Hkv)
        # a bound far above every sequence: many empty tiles
        assert bwd_dq_grid(lib, 64, 32 * L, L, Hq, Hkv, d)[0] is True, (L, Hq, Hkv)
    for S, L, Hq, Hkv, d in [(1, 16384, 32, 32, 128), (1, 8192, 64, 64, 128), (1, 65536, 32, 8, 128), (1, 32768, 32, 8, 128),
                             (4, 2048, 64, 64, 128), (1, 16384, 64, 64, 64), (1, 131072, 12, 2, 128), (1, 16384, 64, 16, 128)]:
        assert bwd_dq_grid(lib, S, S * L, L, Hq, Hkv, d)[0] is True, (S, L, Hq, Hkv)
    for S, tokens, bound, Hq, Hkv, d in [(24, 19500, 1500, 16, 16, 128), (24, 19500, 1500, 40, 20, 128), (32, 19200, 8192, 64, 8, 128),
                                         (8, 8000, 16384, 32, 8, 128), (32, 19200, 8192, 28, 4, 128), (128, 28800, 4096, 28, 4, 128)]:
        assert bwd_dq_grid(lib, S, tokens, bound, Hq, Hkv, d)[0] is True, (S, tokens, bound, Hq, Hkv)
    assert bwd_dq_grid(lib, 1, 300, 65535 * 128, 4, 2, 128)[0] is False
    assert bwd_dq_grid(lib, 1, 300, 65535 * 128 + 1, 4, 2, 128)[0] is True        # beyond the grid's second axis
    for S, tokens, bound, Hq, Hkv in [(65535, 2 ** 31 - 1, 2 ** 31 - 1, 65535, 65535), (65535, 1, 2 ** 31 - 1, 65535, 1), (1, 2 ** 31 - 1, 1, 1, 1)]:
        bwd_dq_grid(lib, S, tokens, bound, Hq, Hkv, 128)                           # (nothing overflows)
