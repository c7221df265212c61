"""The CUDA-core fold's column-sum tiles of a lone product: wide operands are cut
into more tiles than 256 rows make, narrow ones, whose tiles would add to the same
few accumulators, are not.  Read off the workspace, which holds the tile table."""
import numpy as np
import pytest

from paper_2508_21393_gb300 import binding as B


def _bytes(m, k, mont, pad, rows):
    def mat(r, c):
        p = 0 if mont else pad
        return B.vl_mat(1 << 20, r, c, c + p, B.VL_FR_MONT if mont else B.VL_I16, 0, B.VL_DEVICE, 0)
    job = B.vl_job()
    job.P, job.Q = mat(m, k), mat(k, 1)
    o = B.vl_batch_opts()
    o.fold_engine, o.colsum_rows = 1, rows
    n = B.vl_workspace_bytes([job], o)
    assert n > 0
    return n


@pytest.mark.parametrize("m,k", [(1024, 1), (4096, 1), (4096, 5), (4096, 8), (4096, 16), (4096, 64), (16384, 5), (16384, 64),
                                 (300, 8), (1024, 16)])
@pytest.mark.parametrize("mont,pad", [(0, 0), (0, 3), (1, 0)])
def test_narrow_column_sums_keep_their_tiles(m, k, mont, pad):
    if mont and k >= 16:  # one column per thread: sixteen and more columns have few row lanes
        pytest.skip("wide enough for smaller tiles")
    assert _bytes(m, k, mont, pad, 0) == _bytes(m, k, mont, pad, 256)


@pytest.mark.parametrize("m,k,mont", [(601, 2057, 0), (512, 2048, 1), (4096, 1024, 0), (1024, 512, 0), (256, 256, 1)])
def test_wide_column_sums_are_cut(m, k, mont):
    assert _bytes(m, k, mont, 3, 0) > _bytes(m, k, mont, 3, 256)
