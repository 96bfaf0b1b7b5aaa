"""The route of a sector by its size (host arithmetic, no GPU)."""
import os

import pytest


@pytest.fixture(scope="module")
def m():
    import __graft_entry__ as g
    b = g._build_module()
    if not os.path.exists(b.LIB):
        b.build()
    import paper_2303_11409_gb300
    return paper_2303_11409_gb300


SIZES = {"square": lambda k: (k, k), "flat": lambda k: (int(0.85 * k), k), "wide": lambda k: (k, 2 * k),
         "tall": lambda k: (2 * k, k)}


@pytest.mark.parametrize("shape", SIZES)
def test_no_size_falls_out_of_the_block_sweeps(m, shape):
    """One block pair has to fit the shared memory of the FP32 sweeps and of the FP64 sweeps behind them: from 586
    columns there are sizes at which a pair that just fits the first does not fit the second."""
    for k in range(26, 1500):
        rows, cols = SIZES[shape](k)
        plan = m.svd_sector_plan(rows, cols)
        if min(rows, cols) > 24:
            assert plan["path"] == m.MPS_SVD_REFINED, (rows, cols)
        kept = m.svd_sector_plan(rows, cols, keep_phases=True)
        start = m.MPS_SVD_FP32_START if min(rows, cols) >= 192 else 0
        assert kept["path"] == m.MPS_SVD_SWEEPS | start, (rows, cols)


@pytest.mark.parametrize("rows,cols", [(7041, 191), (7041, 192), (7040, 192), (9000, 640), (200, 7100), (7100, 30)])
def test_columns_too_long_for_a_front_keep_the_fp32_start(m, rows, cols):
    """A front copies the QR's reflector, 16 bytes a row, to shared memory (7040 rows)."""
    path = m.svd_sector_plan(rows, cols)["path"]
    if max(rows, cols) <= 7040:
        assert path == m.MPS_SVD_REFINED
    else:
        assert path == m.MPS_SVD_SWEEPS | (m.MPS_SVD_FP32_START if min(rows, cols) >= 192 else 0)


def test_raising_the_fp32_limit_keeps_smaller_sectors_in_fp64(m):
    sizes = [(15, 15), (24, 24), (60, 60), (250, 260), (399, 900), (400, 400), (700, 500)]
    try:
        for k in (1, 64, 192):
            m.svd_mixed_min_k(k)
            assert all(m.svd_sector_plan(*s)["path"] == m.MPS_SVD_REFINED for s in sizes)
            for s in sizes:
                start = m.MPS_SVD_FP32_START if min(s) >= max(k, 96) else 0      # from the block clusters' sizes
                assert m.svd_sector_plan(*s, keep_phases=True)["path"] == m.MPS_SVD_SWEEPS | start
        m.svd_mixed_min_k(400)
        for s in sizes:
            assert m.svd_sector_plan(*s)["path"] == (m.MPS_SVD_REFINED if min(s) >= 400 else m.MPS_SVD_SWEEPS)
        m.svd_mixed_min_k(0)
        for s in sizes:
            assert m.svd_sector_plan(*s)["path"] == m.svd_sector_plan(*s, keep_phases=True)["path"] == m.MPS_SVD_SWEEPS
    finally:
        m.svd_mixed_min_k(192)
