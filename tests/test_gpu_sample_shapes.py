"""Pattern sampling where the columns of a site's products fill less than one warp, several warps and more than the
whole CTA, against a plain walk: the products are laid out over lanes and shared by warps differently in each.

The walk takes the library's own site tensors (FP64 on both sides), so the patterns are the same integers unless a
uniform falls within rounding of a threshold; a conditional probability is a ratio of sums of squares of
at most some hundred rows, off by less than 1e-13 relative, so a pattern's over L sites by less than L 1e-13 < 1e-11.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _draw(sites, d, N, u):
    pat, prob = [], []
    for row in u:
        v, c, p, out = np.ones(1, complex), N, 1.0, []
        for s, x in enumerate(row):
            w = {i: v @ sites[s][(c, c - i)] for i in range(d) if (c, c - i) in sites[s]}
            n2 = {i: float(np.vdot(y, y).real) for i, y in w.items()}
            tot, acc, pick = sum(n2.values()), 0.0, max(n2)
            for i in sorted(n2):
                acc += n2[i] / tot
                if x < acc:
                    pick = i
                    break
            p *= n2[pick] / tot
            v = w[pick] / np.sqrt(n2[pick])
            c -= pick
            out.append(pick)
        pat.append(out)
        prob.append(p)
    return np.array(pat), np.array(prob)


@pytest.mark.parametrize("d, L, layers, chi", [(2, 8, 2, 4), (3, 12, 12, 60), (5, 12, 12, 130), (2, 16, 16, 256),
                                               (8, 8, 8, 700)])
def test_gpu_sampling_over_column_counts(gpu_lib, d, L, layers, chi):
    rng = np.random.default_rng(7)
    occ = [1 if s % 2 == 0 else 0 for s in range(L)] if d == 2 else [1] * L
    g = gpu_lib.MPS(d, occ, chi)
    for r in range(layers):
        for s in range(r % 2, L - 1, 2):
            g.apply_gate2(s, _gate(rng, d), chi, 0.0)
    u = W.uniforms(40, L, seed=3)
    got, prob = g.sample(u)
    ref, pref = _draw([g.site(s) for s in range(L)], d, sum(occ), u)
    assert np.array_equal(got, ref)
    assert np.max(np.abs(prob - pref) / pref) < 1e-11


def _gate(rng, d):
    """A random unitary on each total occupation's states |i, q - i>."""
    def unitary(n):
        return np.linalg.qr(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))[0]
    return [unitary(min(q, d - 1) - max(0, q - d + 1) + 1) for q in range(2 * d - 1)]


@pytest.mark.parametrize("dim", [1400, 1527, 1530, 1536, 1540, 5000])
def test_rows_and_columns_that_just_fill_the_default_shared_memory(gpu_lib, dim):
    """One charge of dim states on two neighbouring bonds: dim rows and dim columns side by side, 16 bytes each, around
    48 KB and well beyond."""
    m = gpu_lib
    rng = np.random.default_rng(dim)
    L, s = 30, 14
    occ = [1, 0] * (L // 2)
    q = [sum(occ[b:]) for b in range(L + 1)]
    g = m.MPS(2, occ, dim)
    for b in (s, s + 1):
        g.set_bond(b, {q[b]: np.ones(dim) / np.sqrt(dim)})
    for x, shape in ((s - 1, (1, dim)), (s, (dim, dim)), (s + 1, (dim, 1))):
        g.set_site(x, {(q[x], q[x + 1]): rng.standard_normal(shape) + 1j * rng.standard_normal(shape)})
    got, prob = g.sample(W.uniforms(5, L, seed=1))
    assert np.array_equal(got, [occ] * 5)
    assert np.max(np.abs(prob - 1.0)) <= 1e-12
    g.close()
