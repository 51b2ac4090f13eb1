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


@pytest.mark.parametrize("sms", [1, 8, 32, 76, 127, 132, 152])
def test_search_shape_fits_on_fewer_sms(sms):
    """The vectors of up to 250000 rows fit in a whole device's shared memory;
    on fewer SMs the steps stream them."""
    for n in (1, 5, 2000, 60000, 131072, 249999, 250000, 250001, 1000000):
        for nhub, nmid in ((0, 0), (n // 100, n // 3), (n // 2, n - n // 2)):
            grid, threads, smem, stream = wl.wl_selftest_search_shape(n, 8 * n, nhub, nmid, sms)
            assert 1 <= grid <= sms and 0 < threads <= 1024 and threads % 32 == 0
            assert 0 <= smem <= SMEM, (n, nhub, nmid, smem)
            if sms == 152:
                assert bool(stream) == (n > 250000)


@pytest.mark.parametrize("fp64", [0, 1])
@pytest.mark.parametrize("n,nnz", [(1, 0), (2000, 20000), (20011, 240000), (10 ** 6, 12 * 10 ** 6), (10 ** 8, 10 ** 9)])
def test_column_blocks_widest_first(fp64, n, nnz):
    """Every column once, widths powers of two up to 64, none wider than the one
    before it (workspaces are sized by the first), a padded block last among its
    width."""
    for k in range(0, 200):
        b = wl.wl_selftest_column_blocks(k, n, nnz, fp64)
        assert sum(kr for _, kr in b) == k
        assert all(K in (1, 2, 4, 8, 16, 32, 64) and 0 < kr <= K for K, kr in b)
        assert all(b[i][0] >= b[i + 1][0] for i in range(len(b) - 1)), (k, b)
        assert all(b[i][1] >= b[i + 1][1] for i in range(len(b) - 1) if b[i][0] == b[i + 1][0]), (k, b)
        assert sum(kr < K for K, kr in b) <= 1
