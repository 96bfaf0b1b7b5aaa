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
