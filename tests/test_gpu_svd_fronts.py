"""Sector SVDs at the sizes where the refined path changes kernel or layout.

Whole refinement inside one CTA (up to 24 columns) with groups of 16 and 32 lanes and columns too long for their
registers; one-CTA fronts (25 columns to what fits shared memory) with groups of 16 and 8 lanes and round-robin
sweeps; cluster fronts whose blocks have equal and unequal lengths, that stay in shared memory and that do
not, with columns held in registers by 16 and 32 lanes and longer ones; tall and wide.

Bounds, for an m x n matrix with N = max(m, n): Householder QR and the products have backward errors of a few
N eps |M|_2, so sigma is within 4 N eps sigma_max; columns are orthogonalised to eps max(n, 32) each, so
Y^dag Y = 1 within 4 eps max(n, 32) + 8 N eps for the vectors above the noise floor, and (M Y)^dag (M Y) = S^2 within
8 N eps sigma_max^2.
"""
import numpy as np
import pytest
import scipy.linalg

import workloads as W

pytestmark = pytest.mark.gpu

EPS = np.finfo(np.float64).eps
SMALL = [(1, 1), (1, 9), (7, 1), (2, 2), (3, 2), (2, 5), (8, 8), (15, 16), (16, 16), (17, 17), (5, 90), (23, 24),
         (24, 24), (24, 70), (90, 24), (6, 180)]
ONE_CTA = [(25, 25), (26, 25), (33, 34), (36, 130), (25, 170), (48, 48), (49, 49), (50, 46), (64, 128), (80, 33), (95, 95),
           (96, 96), (97, 97), (104, 104), (110, 110)]
CLUSTER = [(112, 112), (113, 117), (130, 238), (300, 40), (31, 420), (192, 192), (193, 193), (194, 250), (240, 241),
           (300, 310), (257, 384), (356, 358), (385, 385), (390, 430)]


@pytest.mark.parametrize("decades", [0.0, 8.0])
@pytest.mark.parametrize("shapes", [SMALL, ONE_CTA, CLUSTER], ids=["small", "one-cta", "cluster"])
def test_fronts_match_lapack(gpu_lib, shapes, decades):
    m = gpu_lib
    rng = np.random.default_rng(int(decades) + len(shapes))
    mats = [W.random_complex(s, rng) for s in shapes]
    scales = [np.sort(10.0 ** (-decades * rng.random(s[0])))[::-1].copy() for s in shapes]
    for A, w, (s, y, settled) in zip(mats, scales, m.svd_sectors(mats, rowscales=scales)):
        M = w[:, None] * A
        N = max(M.shape)
        S = scipy.linalg.svd(M, compute_uv=False, lapack_driver="gesvd")
        assert settled >= 0
        assert np.all(np.diff(s) <= 0)
        assert np.max(np.abs(s - S)) <= 4 * N * EPS * S[0], M.shape
        good = s > 64 * N * EPS * S[0]
        Y = y[:, good]
        assert np.max(np.abs(Y.conj().T @ Y - np.eye(Y.shape[1]))) <= 4 * EPS * max(M.shape[1], 32) + 8 * EPS * N, M.shape
        MY = (M / S[0]) @ Y
        assert np.max(np.abs(MY.conj().T @ MY - np.diag((s[good] / S[0]) ** 2))) <= 8 * N * EPS, M.shape


def test_fronts_do_not_depend_on_their_batch(gpu_lib):
    m = gpu_lib
    rng = np.random.default_rng(3)
    mats = [W.random_complex(s, rng) for s in [(20, 22), (60, 60), (120, 112), (193, 193)]]
    every = m.svd_sectors(mats)
    for A, (s, y, _) in zip(mats, every):
        s1, y1, _ = m.svd_sectors([A])[0]
        assert np.array_equal(s, s1) and np.array_equal(y, y1)


def test_fronts_whose_block_pair_just_fits(gpu_lib):
    """Sizes at which a pair of FP32 blocks fits shared memory and the same pair of FP64 blocks would not."""
    m = gpu_lib
    rng = np.random.default_rng(17)
    mats = [W.random_complex(s, rng) for s in [(590, 590), (598, 660), (710, 710)]]
    scales = [np.sort(10.0 ** (-6.0 * rng.random(A.shape[0])))[::-1].copy() for A in mats]
    for A, w, (s, y, steps, path) in zip(mats, scales, m.svd_sectors_path(mats, scales)):
        M = w[:, None] * A
        N = max(M.shape)
        assert path == m.MPS_SVD_REFINED and steps > 0
        S = scipy.linalg.svd(M, compute_uv=False, lapack_driver="gesvd")
        assert np.max(np.abs(s - S)) <= 4 * N * EPS * S[0], M.shape
        Y = y[:, s > 64 * N * EPS * S[0]]
        assert np.max(np.abs(Y.conj().T @ Y - np.eye(Y.shape[1]))) <= 4 * EPS * M.shape[1] + 8 * EPS * N, M.shape
