"""Quasiparticle energies (Cholesky, tridiagonal form, sections on Sturm counts) at the orders
where the number of sections per step changes: one and two rows (64 sections), 4 and 5 (32 and
16), 8 and 9 (16 and 8), 18 and 19 (8 and 4), the largest; matrices that are diagonal, tridiagonal or
a multiple of one already; and a metric that is not positive definite.

Tolerance: with ||X|| <= 4 and a metric between 0.7 and 1.3, backward errors of N eps ||X|| / 0.7
= 80 x 1.1e-16 x 6 < 6e-14; 1e-12 is the bound.
"""
import numpy as np
import pytest

import oracle
from test_gpu_parity import dev
from test_gpu_small_inverse import _inputs, _plan

pytestmark = pytest.mark.gpu


def _check(p, H, Sx, S, om, mu=0.1):
    ref = oracle.qp_energies(H, Sx, S, mu, 20.0, om)
    E = p.qp_energies(dev(H), mu, Sigx_k=dev(Sx), Sig_k_iw=dev(S) if S is not None else None)
    p.sync()
    assert np.abs(E.cpu().numpy().reshape(ref.shape) - ref).max() < 1e-12


@pytest.mark.parametrize("n_atoms,n_orb", [(1, 1), (1, 2), (1, 4), (1, 5), (1, 8), (1, 9), (2, 9), (19, 1), (5, 16)])
def test_orders(n_atoms, n_orb):
    p, tau, om = _plan(n_atoms, n_orb)
    N = n_atoms * n_orb
    H, Sx, S = _inputs(2, len(om), N, 40 + N)
    _check(p, H, Sx, 0.5 * S, om)
    _check(p, H, Sx, None, om)


@pytest.mark.parametrize("n_atoms,n_orb", [(1, 2), (3, 4), (5, 9)])
def test_special_matrices(n_atoms, n_orb):
    p, tau, om = _plan(n_atoms, n_orb)
    N = n_atoms * n_orb
    rng = np.random.default_rng(6)
    t = rng.standard_normal(N - 1) + 1j * rng.standard_normal(N - 1)
    tri = np.diag(rng.standard_normal(N)).astype(np.complex128) + np.diag(t, 1) + np.diag(t.conj(), -1)
    blocks = np.kron(np.eye(N // 2 + 1), np.array([[0.0, 1.0], [1.0, 0.0]]))[:N, :N]  # +-1, many times over
    for a, b in ((np.zeros((N, N)), 0.7 * np.eye(N)), (np.diag(np.arange(N) % 3 - 1.0), tri), (blocks, -blocks)):
        H = np.array([a, b], np.complex128)
        _check(p, H, np.zeros_like(H), None, om)


def test_indefinite_metric():
    """I - S1 negative in one direction at the second momentum only: NaN there, energies at the first."""
    p, tau, om = _plan(1, 6)
    H, Sx, S = _inputs(2, len(om), 6, 3)
    S = 0.2 * S
    i0, i1 = list(om).index(0), list(om).index(1)
    S[1, i1, 2, 2] = S[1, i0, 2, 2] + 1j * (2 * np.pi / 20.0) * 4.0  # S1 = 4 on that diagonal
    E = p.qp_energies(dev(H), 0.1, Sigx_k=dev(Sx), Sig_k_iw=dev(S)).cpu().numpy().reshape(2, 6)
    p.sync()
    ref = oracle.qp_energies(H[:1], Sx[:1], S[:1], 0.1, 20.0, om)
    assert np.isnan(E[1]).all() and np.abs(E[:1] - ref).max() < 1e-12
