"""Host rules that pick a kernel, over ranges of call sizes: the library is asked without a GPU."""
import ctypes

import pytest

from gpu_common import NARROW, UNITS, linear_schedule


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
