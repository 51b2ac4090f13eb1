"""Launch shapes of the cooperative kernels on whole and on smaller devices
(a part of a GPU has fewer SMs, and may place no clusters). No GPU."""
import pytest

from paper_2601_11338_gb300 import wl

SMEM = 227 * 1024


@pytest.mark.parametrize("fp64", [0, 1])
@pytest.mark.parametrize("sms", [1, 8, 16, 76, 152])
def test_cg_shape_without_clusters(fp64, sms):
    for K in (1, 2, 4, 8, 16, 32, 64):
        for n in (1, 2, 33, 257, 1000, 2048, 4096, 8192):
            nnz = 8 * n
            with_c = wl.wl_selftest_cg_shape(fp64, K, n, nnz, 0, 0, sms, True)
            sh = wl.wl_selftest_cg_shape(fp64, K, n, nnz, 0, 0, sms, False)
            if sh is not None:
                grid, threads, smem, cluster = sh
                assert not cluster and 1 <= grid <= sms and threads % 32 == 0 and smem <= SMEM, (K, n, sh)
            elif with_c is not None:  # the grid of a whole device is never smaller than the cluster
                assert sms < 16, (K, n, with_c)
            if with_c is not None and with_c[3]:
                assert with_c[0] <= 16 and with_c[2] <= SMEM
