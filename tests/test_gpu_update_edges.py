"""One two-site update on hand-made blocks, against the oracle: block dimensions at the edges of the 8 x 8 product
tiles and of the 16-deep stages, and selections over more sectors, more values and more equal values than the
selection kernel keeps in shared memory.

Kept dimensions are the same integers.  Schmidt values agree within 1e-12 of the largest (a few N eps for sectors of
some hundred rows), and the gauge-free product B^[s] B^[s+1] within 1e-9 of its largest element: the
kept subspace turns by the SVD's error N eps sigma_max over the gap at the cut, about 1e-13 times 10^3.
"""
import numpy as np
import pytest

from oracle import U1MPS

pytestmark = pytest.mark.gpu


def _update(m, d, L, N, s, tables, chi, rng, values=None):
    """The GPU's and the oracle's state after one random gate on sites (s, s + 1) of random blocks."""
    st = U1MPS.product(d, [N // L + (1 if k < N % L else 0) for k in range(L)])
    for b, t in zip((s, s + 1, s + 2), tables):
        st.bond[b] = dict(t)
        st.lam[b] = {c: np.sort(rng.random(n) + 0.1)[::-1].copy() if values is None else values(n) for c, n in t.items()}
    for k, (left, right) in ((s, tables[:2]), (s + 1, tables[1:])):
        st.B[k] = {(l, r): rng.standard_normal((a, b)) + 1j * rng.standard_normal((a, b))
                   for l, a in left.items() for r, b in right.items() if 0 <= l - r < d}
    g = m.MPS(d, [N // L + (1 if k < N % L else 0) for k in range(L)], max(chi, max(sum(t.values()) for t in tables)))
    for b in (s, s + 1, s + 2):
        g.set_bond(b, st.lam[b])
    for k in (s, s + 1):
        g.set_site(k, st.B[k])
    gate = []
    for q in range(2 * d - 1):
        n = min(q, d - 1) - max(0, q - d + 1) + 1
        gate.append(np.linalg.qr(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))[0])
    g.apply_gate2(s, gate, chi, 0.0)
    st.apply_gate2(s, gate, chi, 0.0)
    return g, st


def _same(g, st, s, d):
    lam, ref = g.bond(s + 1), st.lam[s + 1]
    assert {c: len(v) for c, v in lam.items()} == {c: len(v) for c, v in ref.items()}
    top = max(v[0] for v in ref.values())
    assert max(np.max(np.abs(lam[c] - ref[c])) for c in ref) <= 1e-12 * top
    A, B = g.site(s), g.site(s + 1)

    def product(A, B):
        out = {}
        for (l, c), a in A.items():
            for (c2, r), b in B.items():
                if c2 == c:
                    key = (l, c, r)
                    out[key] = a @ b
        return out
    got, want = product(A, B), product(st.B[s], st.B[s + 1])
    assert got.keys() == want.keys()
    big = max(np.max(np.abs(x)) for x in want.values())
    assert max(np.max(np.abs(got[k] - want[k])) for k in want) <= 1e-9 * big


@pytest.mark.parametrize("dims", [(1, 7, 8, 9, 1), (8, 15, 16, 17, 3), (16, 24, 25, 1, 33), (2, 40, 7, 64, 5)])
@pytest.mark.parametrize("part", [1.0, 0.4])
def test_update_at_tile_edges(gpu_lib, dims, part):
    rng = np.random.default_rng(sum(dims))
    d, L, N, s = 3, 12, 12, 5
    tables = [{4 + k: dims[(k + j) % 5] for k in range(5)} for j in range(3)]
    tables = [{c - (1 if j == 2 else 0): n for c, n in t.items()} for j, t in enumerate(tables)]
    chi = max(1, int(part * sum(tables[1].values())))
    g, st = _update(gpu_lib, d, L, N, s, tables, chi, rng)
    _same(g, st, s, d)


@pytest.mark.parametrize("dim, chi", [(1, 300), (2, 150)])
def test_selection_over_more_sectors_than_a_table(gpu_lib, dim, chi):
    """281 charges on the middle bond (d = 8, L = 80): more sectors than the selection stages at once."""
    rng = np.random.default_rng(dim)
    tables = [{c: dim for c in range(lo, hi)} for lo, hi in ((7, 281), (0, 281), (0, 274))]
    g, st = _update(gpu_lib, 8, 80, 280, 39, tables, chi, rng)
    _same(g, st, 39, 8)


def test_selection_over_more_values_than_a_table(gpu_lib):
    """About 5000 singular values in 11 sectors."""
    rng = np.random.default_rng(5)
    tables = [{c: 230 for c in range(lo, lo + 10)} for lo in (9, 8, 7)]
    g, st = _update(gpu_lib, 3, 24, 24, 11, tables, 900, rng)
    _same(g, st, 11, 3)


@pytest.mark.parametrize("dim, charges, chi", [(40, 11, 100), (150, 11, 700), (300, 11, 2000), (600, 9, 2500), (2, 281, 401)])
def test_selection_among_equal_values(gpu_lib, dim, charges, chi):
    """Unitary blocks between equal charges and equal Schmidt values: Theta'(c) is a product of unitaries, the values of
    all sectors are equal up to rounding, and the ties go to the sectors in ascending order until chi are kept (up to
    and past the values and the sectors that are staged in shared memory)."""
    m = gpu_lib
    rng = np.random.default_rng(dim)
    d, L = 2, 2 * charges + 20
    s = L // 2 - 1
    st = U1MPS.product(d, [k % 2 for k in range(L)])
    table = {5 + q: dim for q in range(charges)}
    for b in (s, s + 1, s + 2):
        st.bond[b] = dict(table)
        st.lam[b] = {c: np.ones(dim) / np.sqrt(dim * charges) for c in table}
    for k in (s, s + 1):
        st.B[k] = {(c, r): np.zeros((dim, dim), complex) for c in table for r in table if 0 <= c - r < d}
        for c in table:
            st.B[k][(c, c)] = np.linalg.qr(rng.standard_normal((dim, dim)) + 1j * rng.standard_normal((dim, dim)))[0]
    g = m.MPS(d, [k % 2 for k in range(L)], max(chi, dim * charges))
    for b in (s, s + 1, s + 2):
        g.set_bond(b, st.lam[b])
    for k in (s, s + 1):
        g.set_site(k, st.B[k])
    gate = [np.eye(1, dtype=complex), np.eye(2, dtype=complex), np.eye(1, dtype=complex)]
    g.apply_gate2(s, gate, chi, 1e-10)
    kept = {c: len(v) for c, v in g.bond(s + 1).items()}
    want, left = {}, chi
    for c in table:
        if left > 0:
            want[c] = min(dim, left)
            left -= want[c]
    assert kept == want
    for c, v in g.bond(s + 1).items():
        assert np.max(np.abs(v - 1 / np.sqrt(chi))) <= 1e-12


@pytest.mark.parametrize("cutoff", [0.0, -0.0])
def test_a_cutoff_of_minus_zero_is_zero(gpu_lib, cutoff):
    """Values of exactly 0 (empty rows and columns) are not kept by either."""
    m = gpu_lib
    d, L, s, dim = 2, 12, 5, 8
    table = {3: dim, 2: dim}
    g = m.MPS(d, [k % 2 for k in range(L)], 64)
    rng = np.random.default_rng(3)
    for b in (s, s + 1, s + 2):
        g.set_bond(b, {c: np.ones(dim) / np.sqrt(2 * dim) for c in table})
    B = {(c, r): np.zeros((dim, dim), complex) for c in table for r in table if 0 <= c - r < d}
    for c in table:
        B[(c, c)][:3, :3] = rng.standard_normal((3, 3))
    for k in (s, s + 1):
        g.set_site(k, B)
    g.apply_gate2(s, [np.eye(1, dtype=complex), np.eye(2, dtype=complex), np.eye(1, dtype=complex)], 64, cutoff)
    assert {c: len(v) for c, v in g.bond(s + 1).items()} == {2: 3, 3: 3}
    assert all(np.all(v > 0) for v in g.bond(s + 1).values())
