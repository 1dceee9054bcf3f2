"""Host rules that pick a kernel, over ranges of call sizes: the library is asked without a GPU."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def lib():
    from paper_2609_35140_b200 import binding
    lib = binding.load()
    lib.tik_selftest_decode_cluster.argtypes = [ctypes.c_int64] + 4 * [ctypes.c_int]
    return lib


@pytest.mark.parametrize("max_clusters", [0, 1, 33, 37])
def test_clusters_only_while_all_of_them_run_at_once(lib, max_clusters):
    """A cluster decode whose clusters do not all fit takes a second wave: 1.5 to 2 times the time of the kernels
    without clusters.  How many fit is the device's answer (33 of four CTAs on 148 SMs), not SMs / 4."""
    for chunks in range(1, 60):
        got = lib.tik_selftest_decode_cluster(chunks, 4000, 8, 128, max_clusters)
        assert got == (4 if chunks <= max_clusters else 0), chunks
    for refused in ((4, 896, 8, 128), (4, 4000, 9, 128), (4, 4000, 8, 64)):
        assert lib.tik_selftest_decode_cluster(*refused, max_clusters) == 0
