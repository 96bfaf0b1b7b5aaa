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


@pytest.mark.parametrize("decades", [0.0, 8.0])
def test_sweeps_of_reduced_precision_updates_match_lapack(gpu_lib, decades):
    """Pivoted QR and FP64 sweeps in one CTA (up to about 95 columns) and on clusters, from 192 columns behind FP32
    sweeps and a Cholesky QR of their rotations."""
    m = gpu_lib
    shapes = [(15, 16), (48, 48), (95, 95), (112, 112), (130, 238), (192, 192), (193, 193), (257, 255), (300, 310),
              (420, 260), (230, 480), (640, 610)]
    mats, scales = _graded(shapes, decades, 21 + int(decades))
    for A, w, (s, y, sweeps, path) in zip(mats, scales, m.svd_sectors_path(mats, scales, keep_phases=True)):
        start = m.MPS_SVD_FP32_START if min(A.shape) >= 192 else 0
        assert path == m.MPS_SVD_SWEEPS | start and sweeps > 0
        _check(w[:, None] * A, s, y)


def test_which_sectors_are_refined(gpu_lib):
    """Spectra without large degenerate groups settle at every size; large groups of equal values and zero matrices
    are left to the FP64 sweeps."""
    m = gpu_lib
    from tests import test_gpu_svd_fronts as F
    from tests import test_gpu_svd_refine as T
    for decades in (0.0, 8.0):
        mats, scales = _graded(T.SHAPES + F.SMALL + F.ONE_CTA + F.CLUSTER, decades, 5)
        assert all(r[3] == m.MPS_SVD_REFINED for r in m.svd_sectors_path(mats, scales))
    rng = np.random.default_rng(7)
    Q, P = W.haar_unitary(72, rng), W.haar_unitary(72, rng)
    left = [Q @ np.diag(np.repeat([1.0, 0.5, 0.25], 24)) @ P,
            Q @ np.diag(np.concatenate([1 + 1e-10 * np.arange(36), 0.2 + 1e-5 * np.arange(36)])) @ P,
            np.zeros((50, 60), complex)]
    settled = [W.random_complex((80, 13), rng) @ W.random_complex((13, 70), rng), np.eye(64, dtype=complex),
               1e-130 * W.random_complex((50, 50), rng), W.haar_unitary(300, rng)]
    swept = m.MPS_SVD_SWEEPS | m.MPS_SVD_FP32_START
    assert [r[3] for r in m.svd_sectors_path(left)] == [swept, swept, m.MPS_SVD_SWEEPS]
    assert [r[3] for r in m.svd_sectors_path(settled)] == [m.MPS_SVD_REFINED] * len(settled)


@pytest.mark.parametrize("L,chi", [(10, 300), (12, 700)])
def test_when_teams_are_formed(gpu_lib, L, chi):
    """Few large sectors of a TF32 update take teams of CTAs, unless the phases are captured; an FP64 update's are refined,
    but for those up to 24 columns that one CTA cannot hold (13 x 522 here)."""
    import torch
    from oracle import gates
    from tests.helpers import load_state, random_state
    m = gpu_lib
    st = random_state(L, 5, L, chi, seed=chi)
    stream = torch.cuda.Stream()
    for precision, graphs in ((m.MPS_TF32, False), (m.MPS_TF32, True), (m.MPS_FP64, False)):
        g = m.MPS(5, [1] * L, chi, precision=precision, stream=stream.cuda_stream)
        load_state(g, st)
        g.set_graphs(graphs)
        s = L // 2 - 1
        g.apply_gate2(s, gates.bh_gate(L, s, 5, 1.0, 2.0, 0.3), chi, 1e-10)
        p = g.last_batch_paths()
        if precision == m.MPS_FP64:
            assert p["refined"] >= 10 and p["swept"] <= 1 and p["fp32_start"] == p["on_teams"] == 0
        else:
            assert p["refined"] == 0 and p["swept"] > 0 and (p["on_teams"] > 0) == (not graphs)
        g.close()


@pytest.mark.parametrize("min_k", [0, 16])
def test_small_sectors_on_one_cta_and_on_block_clusters(gpu_lib, min_k):
    m = gpu_lib
    mats, scales = _graded([(16, 16), (17, 40), (48, 48), (64, 31), (85, 85), (90, 120), (130, 70)], 8.0, 31)
    try:
        m.svd_cluster_min_k(min_k)
        out = m.svd_sectors_path(mats, scales, keep_phases=True)
    finally:
        m.svd_cluster_min_k(0)
    for A, w, (s, y, sweeps, path) in zip(mats, scales, out):
        assert path == m.MPS_SVD_SWEEPS and sweeps > 0
        _check(w[:, None] * A, s, y)


def test_expired_staging_waits_end_the_call_with_a_status(gpu_lib):
    """FP64 sweeps, FP32 sweeps ahead of them, and a sector of one CTA, which stages nothing."""
    m = gpu_lib
    mats, scales = _graded([(112, 112), (300, 310), (48, 48)], 4.0, 41)
    m.svd_inject_stall(1)
    try:
        out = m.svd_sectors_path(mats, scales, keep_phases=True)
    finally:
        m.svd_inject_stall(0)
    assert [r[2] for r in out[:2]] == [-2, -2] and [r[3] for r in out[:2]] == [0, 0]
    assert out[2][2] > 0 and out[2][3] == m.MPS_SVD_SWEEPS
    for A, w, (s, y, sweeps, path) in zip(mats, scales, m.svd_sectors_path(mats, scales, keep_phases=True)):
        assert sweeps > 0
        _check(w[:, None] * A, s, y)


@pytest.mark.parametrize("graphs", [False, True])
def test_expired_staging_waits_of_an_update_leave_the_state(gpu_lib, graphs):
    """With graphs off the large sectors are on teams of CTAs, with graphs on clusters."""
    import torch
    from oracle import gates
    from tests.helpers import load_state, random_state
    m = gpu_lib
    L, chi, s = 10, 300, 4
    stream = torch.cuda.Stream()
    g = m.MPS(5, [1] * L, chi, precision=m.MPS_BF16X3, stream=stream.cuda_stream)
    load_state(g, random_state(L, 5, L, chi, seed=1))
    g.set_graphs(graphs)
    G = gates.bh_gate(L, s, 5, 1.0, 2.0, 0.3)
    before = [g.bond(s + 1), g.site(s), g.site(s + 1)]
    m.svd_inject_stall(1)
    try:
        with pytest.raises(m.MPSError) as e:
            g.apply_gate2(s, G, chi, 1e-10)
        assert e.value.code == m.MPS_ETIMEOUT
    finally:
        m.svd_inject_stall(0)
    for a, b in zip(before, [g.bond(s + 1), g.site(s), g.site(s + 1)]):
        assert a.keys() == b.keys() and all(np.array_equal(a[k], b[k]) for k in a)
    g.apply_gate2(s, G, chi, 1e-10)
    assert abs(sum(float(np.sum(v ** 2)) for v in g.bond(s + 1).values()) - 1.0) < 1e-12
    g.close()


def test_expired_staging_waits_of_dmrg(gpu_lib):
    from tests.helpers import load_state, random_state
    m = gpu_lib
    L, chi = 10, 300
    terms = m.models.chain_bond_terms("bh", L, 5, J=1.0, U=2.0)
    g = m.MPS(5, [1] * L, chi)
    load_state(g, random_state(L, 5, L, chi, seed=2))
    m.svd_mixed_min_k(0)
    m.svd_inject_stall(1)
    try:
        with pytest.raises(m.MPSError) as e:
            g.dmrg(terms, 1, chi, 1e-12)
        assert e.value.code == m.MPS_ETIMEOUT
    finally:
        m.svd_inject_stall(0)
        m.svd_mixed_min_k(192)
    g.close()
    with pytest.raises(m.MPSError):
        m.svd_inject_stall(64)


def test_expired_waits_of_the_fp32_sweeps_leave_the_sector_to_the_fp64_sweeps(gpu_lib):
    """Fronts on clusters, with blocks that stay in shared memory and that do not; a one-CTA front stages nothing."""
    import time
    m = gpu_lib
    mats, scales = _graded([(130, 238), (240, 241), (257, 384), (390, 430), (112, 112)], 4.0, 43)
    clean = m.svd_sectors_path(mats, scales)
    assert all(r[3] == m.MPS_SVD_REFINED for r in clean)
    m.svd_inject_stall(2)
    try:
        t0 = time.perf_counter()
        out = m.svd_sectors_path(mats, scales)
        took = time.perf_counter() - t0
    finally:
        m.svd_inject_stall(0)
    assert [r[3] for r in out] == [m.MPS_SVD_SWEEPS] * 4 + [m.MPS_SVD_REFINED]
    assert took < 2.0      # one wait of 50 ms a CTA and another for its copies, not one a round
    for A, w, (s, y, sweeps, path) in zip(mats, scales, out):
        assert sweeps > 0
        _check(w[:, None] * A, s, y)
    for (s, y, _, _), (s1, y1, _, _) in zip(clean, m.svd_sectors_path(mats, scales)):
        assert np.array_equal(s, s1) and np.array_equal(y, y1)


def test_columns_too_long_for_a_front(gpu_lib):
    m = gpu_lib
    mats, scales = _graded([(7100, 195), (7100, 40)], 3.0, 47)
    out = m.svd_sectors_path(mats, scales)
    assert [r[3] for r in out] == [m.MPS_SVD_SWEEPS | m.MPS_SVD_FP32_START, m.MPS_SVD_SWEEPS]
    for A, w, (s, y, sweeps, path) in zip(mats, scales, out):
        assert sweeps > 0
        _check(w[:, None] * A, s, y)


@pytest.mark.parametrize("group", [2, 3, 8, 24])
def test_degenerate_values_go_on_from_the_fp32_rotations(gpu_lib, group):
    """Values in equal groups over four decades, which the refinement leaves: one-CTA fronts, cluster fronts, wide and tall.
    The FP64 sweeps start from the front's QR and rotations, so they are few."""
    m = gpu_lib
    rng = np.random.default_rng(group)
    mats = []
    for a, b in [(72, 72), (30, 96), (150, 144), (120, 200), (300, 300), (260, 420), (420, 240), (200, 210)]:
        k = min(a, b)
        v = np.repeat(10.0 ** (-4.0 * np.arange(-(-k // group)) * group / k), group)[:k]
        mats.append((W.haar_unitary(a, rng)[:, :k] * v) @ W.haar_unitary(b, rng)[:k])
    swept = m.MPS_SVD_SWEEPS | m.MPS_SVD_FP32_START
    out = m.svd_sectors_path(mats)
    assert sum(r[3] == swept for r in out) >= 6
    for A, (s, y, steps, path) in zip(mats, out):
        assert path in (swept, m.MPS_SVD_REFINED) and steps > 0
        _check(A, s, y)
