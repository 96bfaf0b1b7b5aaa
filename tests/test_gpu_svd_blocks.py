"""The block-Jacobi sweeps on staged columns (FP64, and FP32 ahead of them), which TF32 and BF16x3 updates run and
which take what the refinement of the other sectors leaves.

Bounds, for an m x n matrix with N = max(m, n): Householder QR and the rotations have backward errors of a few
N eps |M|_2, so sigma is within 4 N eps sigma_max; the sweeps end when every pair of columns is orthogonal to
eps max(n, 32), so Y^dag Y = 1 within 4 eps max(n, 32) + 8 N eps for the vectors above the noise floor, and
(M Y)^dag (M Y) = S^2 within 8 N eps sigma_max^2.
"""
import numpy as np
import pytest
import scipy.linalg

import workloads as W

pytestmark = pytest.mark.gpu

EPS = np.finfo(np.float64).eps


def _graded(shapes, decades, seed):
    rng = np.random.default_rng(seed)
    return ([W.random_complex(s, rng) for s in shapes],
            [np.sort(10.0 ** (-decades * rng.random(s[0])))[::-1].copy() for s in shapes])


def _check(M, s, y):
    N = max(M.shape)
    S = scipy.linalg.svd(M, compute_uv=False, lapack_driver="gesvd")
    assert np.all(np.diff(s) <= 0)
    assert np.max(np.abs(s - S)) <= 4 * N * EPS * S[0], M.shape
    good = s > 64 * N * EPS * S[0]
    Y = y[:, good]
    assert np.max(np.abs(Y.conj().T @ Y - np.eye(Y.shape[1]))) <= 4 * EPS * max(M.shape[1], 32) + 8 * EPS * N, M.shape
    MY = (M / S[0]) @ Y
    assert np.max(np.abs(MY.conj().T @ MY - np.diag((s[good] / S[0]) ** 2))) <= 8 * N * EPS, M.shape


def test_staged_blocks_give_the_same_bits_each_time(gpu_lib):
    """One to seven chunks of block pairs a round pass through the same shared memory, written by the rotations and
    read by the bulk copies."""
    m = gpu_lib
    mats, scales = _graded([(610, 640), (420, 400), (230, 480), (150, 140)], 6.0, 11)
    try:
        m.svd_mixed_min_k(0)
        first, *others = [m.svd_sectors(mats, rowscales=scales) for _ in range(3)]
    finally:
        m.svd_mixed_min_k(192)
    for A, w, (s, y, sweeps) in zip(mats, scales, first):
        assert sweeps > 0
        _check(w[:, None] * A, s, y)
    for out in others:
        for (s, y, _), (s1, y1, _) in zip(first, out):
            assert np.array_equal(s, s1) and np.array_equal(y, y1)
