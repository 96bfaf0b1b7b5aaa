"""The Krylov exponential of TDVP over both of its forms: Taylor steps for short spans |tau| rho, eigenpairs for long ones.

On two sites a TDVP step is the exact evolution of the pair (the Krylov space is the whole charge sector, 5 states here),
so every amplitude equals exp(-i H dt) applied to the start vector.  Both forms round like the phases dt lambda: up to
1600 times a few eps, so 1e-10 leaves two decades.
"""
import itertools

import numpy as np
import pytest

from oracle import dense

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt", [0.01, 3.0, 30.0, 55.0, 80.0, 400.0, -120.0])
def test_two_site_step_is_the_exact_exponential(gpu_lib, dt):
    m = gpu_lib
    d, J, U = 5, 1.0, 2.0
    g = m.MPS(d, [3, 1], 64)
    g.tdvp(m.models.chain_bond_terms("bh", 2, d, J=J, U=U), 1, dt, 64, 0.0)
    H = dense.bh_two_site(d, J, U, 1.0, 1.0)
    psi0 = np.zeros(d * d, dtype=np.complex128)
    psi0[3 * d + 1] = 1.0
    w, v = np.linalg.eigh(H)
    psi = v @ (np.exp(-1j * dt * w) * (v.conj().T @ psi0))
    cfgs = [c for c in itertools.product(range(d), repeat=2) if sum(c) == 4]
    amp = g.amplitudes(cfgs)
    assert np.max(np.abs(amp - psi[[a * d + b for a, b in cfgs]])) <= 1e-10
    g.close()


def test_krylov_vectors_longer_than_one_chunk_a_cta(gpu_lib):
    """<H_eff> before each step of a TDVP sweep, on vectors of 25 to 1.6 million elements: the longest ones pass
    through the Gram-Schmidt kernels in several chunks a CTA (from 622,592 elements).  The energy is the first Lanczos
    scalar of each step, so it shows every sum of a step; the projected evolution conserves it up to the truncated
    weight, of order (dt |H|)^2 relative to the energies' scale |H| of about 30: 1e-5 of it at dt = 1e-4."""
    from tests.helpers import load_state, random_state
    m = gpu_lib
    L, chi = 14, 1700
    terms = m.models.chain_bond_terms("bh", L, 5, J=1.0, U=4.0)
    g = m.MPS(5, [1] * L, chi)
    load_state(g, random_state(L, 5, L, chi, seed=3))
    g.dmrg(terms, 1, chi, 0.0, lanczos_dim=2, tol=1e6)      # one sweep makes the state canonical
    longest = 0
    for s in range(L - 1):
        left, right = g.bond_dims(s), g.bond_dims(s + 2)
        longest = max(longest, sum(a * b for x, a in left.items() for y, b in right.items() if 0 <= x - y <= 8))
    assert longest > 622592
    E = g.tdvp(terms, 1, 1e-4, chi, 0.0, krylov_dim=5)
    assert np.ptp(E) <= 3e-4, E
    for b in (1, L // 2, L - 1):
        assert abs(sum(float(v @ v) for v in g.bond(b).values()) - 1.0) <= 1e-12
