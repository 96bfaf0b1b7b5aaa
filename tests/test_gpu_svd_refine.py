"""Sector SVDs that go through the FP32 Jacobi start and the tensor-core refinement.

Singular values against LAPACK and the right vectors' properties at the sizes where the path can go
wrong: the smallest refined sector, edges of the 64 x 32 product tiles and of the 32-deep stages,
wide and tall sectors, rows graded over many decades, and spectra the refinement must hand to the FP64
sweeps (exactly degenerate, rank deficient, zero, out of the range of squares).

Bounds, for an m x n matrix with N = max(m, n): Householder QR and the products have backward errors
of a few N eps |M|_2, so sigma is within 4 N eps sigma_max; columns are orthogonalised to eps max(n, 32)
each, so Y^dag Y = 1 within 4 eps max(n, 32) for the vectors above the noise floor, and
(M Y)^dag (M Y) = S^2 within 8 N eps sigma_max^2.
"""
import numpy as np
import pytest
import scipy.linalg

import workloads as W

pytestmark = pytest.mark.gpu

EPS = np.finfo(np.float64).eps
SHAPES = [(48, 48), (49, 63), (64, 64), (65, 96), (97, 64), (96, 129), (128, 128), (160, 161), (193, 48), (48, 260),
          (257, 255), (320, 70), (66, 500)]


def _check(M, s, y, settled):
    N = max(M.shape)
    S = scipy.linalg.svd(M, compute_uv=False, lapack_driver="gesvd")
    top = S[0]
    assert np.all(np.diff(s) <= 0)
    assert np.max(np.abs(s - S)) <= 4 * N * EPS * top
    good = s > 64 * N * EPS * top
    Y = y[:, good]
    assert np.max(np.abs(Y.conj().T @ Y - np.eye(Y.shape[1]))) <= 4 * EPS * max(M.shape[1], 32) + 8 * EPS * N
    MY = (M / top) @ Y
    assert np.max(np.abs(MY.conj().T @ MY - np.diag((s[good] / top) ** 2))) <= 8 * N * EPS
    assert settled >= 0


@pytest.mark.parametrize("decades", [0.0, 5.0, 11.0])
def test_refined_sectors_match_lapack(gpu_lib, decades):
    m = gpu_lib
    rng = np.random.default_rng(int(decades) + 40)
    mats = [W.random_complex(s, rng) for s in SHAPES]
    scales = [np.sort(10.0 ** (-decades * rng.random(s[0])))[::-1].copy() for s in SHAPES]
    for A, w, (s, y, st) in zip(mats, scales, m.svd_sectors(mats, rowscales=scales)):
        _check(w[:, None] * A, s, y, st)


def test_spectra_the_refinement_does_not_settle(gpu_lib):
    m = gpu_lib
    rng = np.random.default_rng(7)
    Q, P = W.haar_unitary(72, rng), W.haar_unitary(72, rng)
    blocks = Q @ np.diag(np.repeat([1.0, 0.5, 0.25], 24)) @ P                     # exactly degenerate
    close = Q @ np.diag(np.concatenate([1 + 1e-10 * np.arange(36), 0.2 + 1e-5 * np.arange(36)])) @ P
    rank = W.random_complex((80, 13), rng) @ W.random_complex((13, 70), rng)
    holes = W.random_complex((70, 60), rng)
    holes[:, 11:37] = 0.0
    small, large = 1e-130 * W.random_complex((50, 50), rng), 1e130 * W.random_complex((50, 50), rng)
    mats = [blocks, close, rank, holes, np.eye(64, dtype=complex), small, large, np.zeros((50, 60), complex)]
    out = m.svd_sectors(mats)
    for A, (s, y, st) in zip(mats[:-1], out[:-1]):
        _check(A, s, y, st)
    assert not np.any(out[-1][0]) and not np.any(out[-1][1])


def test_refined_sectors_do_not_depend_on_their_batch(gpu_lib):
    m = gpu_lib
    rng = np.random.default_rng(9)
    mats = [W.random_complex(s, rng) for s in [(70, 90), (130, 64), (20, 20), (200, 210)]]
    every = m.svd_sectors(mats)
    for A, (s, y, _) in zip(mats, every):
        s1, y1, _ = m.svd_sectors([A])[0]
        assert np.array_equal(s, s1) and np.array_equal(y, y1)


@pytest.mark.parametrize("L,chi", [(10, 300), (12, 700)])
def test_teams_give_the_bits_of_the_clusters(gpu_lib, L, chi):
    """A TF32 update whose few large sectors run on teams of CTAs equals, bit for bit, the same update
    with captured phases (which keep the cluster kernels)."""
    import torch
    from oracle import gates
    from tests.helpers import load_state, random_state
    m = gpu_lib
    st = random_state(L, 5, L, chi, seed=chi)
    stream = torch.cuda.Stream()
    out = []
    for graphs in (False, True):
        g = m.MPS(5, [1] * L, chi, precision=m.MPS_TF32, stream=stream.cuda_stream)
        load_state(g, st)
        g.set_graphs(graphs)
        for s in (L // 2 - 1, L // 2, L // 2 - 1):
            g.apply_gate2(s, gates.bh_gate(L, s, 5, 1.0, 2.0, 0.3), chi, 1e-10)
        out.append([g.bond(b) for b in range(L + 1)] + [g.site(s) for s in range(L)])
        g.close()
    for a, b in zip(*out):
        assert a.keys() == b.keys()
        assert all(np.array_equal(a[k], b[k]) for k in a)


def test_more_sectors_than_a_grid_has_rows(gpu_lib):
    """70,000 refined sectors in one call; those on both sides of 65,535 against LAPACK."""
    m = gpu_lib
    rng = np.random.default_rng(70)
    n, k = 70000, 25
    A = rng.standard_normal((n, k, k)) + 1j * rng.standard_normal((n, k, k))
    out = m.svd_sectors_path(list(A))
    assert all(r[3] == m.MPS_SVD_REFINED for r in out)
    for i in [0, 1, *range(65530, 65540), n - 1, *rng.integers(0, n, 200)]:
        _check(A[i], *out[i][:3])


def test_captured_layer_with_every_kind_of_front(gpu_lib):
    """A layer whose sectors take clusters of 8, smaller clusters, one CTA and the whole refinement in one CTA, on side
    streams and behind one another: with captured phases the same bits as without, call after call."""
    import torch
    from oracle import gates
    from tests.helpers import load_state, random_state
    m = gpu_lib
    L, chi, sites = 14, 700, [2, 4, 6, 8, 10]
    st = random_state(L, 5, L, chi, seed=8)
    stream = torch.cuda.Stream()
    out = []
    for graphs in (False, True):
        g = m.MPS(5, [1] * L, chi, stream=stream.cuda_stream)
        load_state(g, st)
        g.set_graphs(graphs)
        for _ in range(3):
            g.apply_layer(sites, [gates.bh_gate(L, s, 5, 1.0, 2.0, 0.1) for s in sites], chi, 1e-10)
            assert g.last_batch_paths()["refined"] > 30
        out.append([g.bond(b) for b in range(L + 1)] + [g.site(s) for s in range(L)])
        if graphs:
            assert g.graph_stats()["launches"] >= 6
        g.close()
    plans = [m.svd_sector_plan(*s) for s in ((300, 300), (130, 140), (60, 60), (20, 20))]
    assert [p["ctas"] for p in plans] == [8, 4, 1, 1], plans
    for a, b in zip(*out):
        assert a.keys() == b.keys()
        assert all(np.array_equal(a[k], b[k]) for k in a)
