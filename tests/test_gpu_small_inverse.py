"""The batched FP64 inverse in shared memory and the particle number from Hessenberg forms,
at the orders where their loops change shape: one and two rows, about a warp, the largest
order held in shared memory and the first one beyond it, against torch's complex128 inverse.

Tolerance: with |w| >= pi / 20 and |M| <= 20 the condition of every matrix is below 130, so an
inverse is good to N eps kappa < 2e-12 and the inverse transform (condition below 100)
to 2e-10 of the largest value; the parity bar of 1e-10 in the Frobenius norm is kept.  N(mu)
is a trace of the same rounding, and the slope of N is at least 1 per Ha around the root, so
mu is compared to 1e-9 as in the Dyson tests.
"""
import numpy as np
import pytest

import oracle
import synth
from test_gpu_parity import TOL, dev, host, rel

pytestmark = pytest.mark.gpu


def _plan(n_atoms, n_orb, kmesh=(2, 1, 1), beta=20.0, n_tau=10):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1911_05633_gb300 import gw
    lat = np.eye(3) * 6.0 * n_atoms
    frac = np.array([[i / n_atoms, 0.0, 0.0] for i in range(n_atoms)])
    om, nu = synth.matsubara_sets(n_tau)
    tau = synth.tau_nodes(beta, n_tau)
    C = np.ones((1, n_orb, n_orb))
    return gw.Plan(lat, frac, np.zeros(n_atoms, np.int32), [n_orb], [1], [C], kmesh, beta, tau, om, nu, 7.0), tau, om


def _inputs(nk, n_w, N, seed):
    rng = np.random.default_rng(seed)
    z = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)
    herm = lambda x: 0.5 * (x + np.conj(np.swapaxes(x, -1, -2)))
    H = herm(z(nk, N, N)) / np.sqrt(N)
    Sx = 0.1 * herm(z(nk, N, N)) / np.sqrt(N)
    S = 0.05 * z(nk, n_w, N, N) / np.sqrt(N)
    return H, Sx, 0.5 * (S + np.conj(np.swapaxes(S[:, ::-1], -1, -2)))


@pytest.mark.parametrize("n_atoms,n_orb", [(1, 1), (1, 2), (1, 3), (3, 11), (8, 9), (8, 14), (9, 13), (9, 16)])
def test_inverse_and_particle_number(n_atoms, n_orb):
    p, tau, om = _plan(n_atoms, n_orb)
    N = n_atoms * n_orb
    H, Sx, S = _inputs(2, len(om), N, N)
    T = p.transform_matrix("F", "iw_to_tau")
    G = lambda mu: oracle.green_iw_to_tau(oracle.dyson_green_iw(H, Sx, S, mu, 20.0, om), H, Sx, mu, 20.0, tau, om, T)
    got = host(p.dyson_green_tau(dev(H), 0.1, Sigx_k=dev(Sx), Sig_k_iw=dev(S)))
    p.sync()
    assert rel(got, G(0.1).reshape(-1)) < TOL
    mu, n = p.chemical_potential(dev(H), float(N), -4.0, 4.0, tol=1e-11, Sigx_k=dev(Sx), Sig_k_iw=dev(S))
    # half filling: N(mu) of the oracle's own solve at that mu, and a sign change around it
    count = lambda m: -2.0 * np.trace(G(m)[:, -1], axis1=1, axis2=2).real.mean()
    assert abs(n - count(mu)) < 1e-9 * N
    assert count(mu - 1e-7) < N < count(mu + 1e-7)


def test_singular_shift_is_still_reported():
    """mu + M exactly singular at the first midpoint of the search: the solve decides, as for any mu."""
    from paper_1911_05633_gb300 import gw
    p, tau, om = _plan(1, 2)
    w = (2 * om + 1) * np.pi / 20.0
    S = np.zeros((2, len(om), 2, 2), np.complex128)
    S[:] = (1j * w)[None, :, None, None] * np.eye(2)  # i w - Sigma = 0
    H = np.zeros((2, 2, 2))
    H[:, 1, 1] = 0.5
    with pytest.raises(gw.GwError) as e:
        p.chemical_potential(dev(H), 2.0, -1.0, 1.0, Sig_k_iw=dev(S))
    assert e.value.status == 6


def test_dyson_inverses_beyond_shared_memory_go_by_columns():
    """Order 117, the first cell here that does not fit, against torch's inverse (as above)."""
    p, tau, om = _plan(9, 13)
    H, Sx, S = _inputs(2, len(om), 117, 5)
    p.timing_enable(True)
    A = p.spectral_function(dev(H), [0.1, 0.3], 0.2, 0.0)
    assert "k_gj_inverse" in p.timing_read() and "k_gj_inverse_blocked" not in p.timing_read()
    z = np.array([0.1, 0.3])[None, :, None, None] + 0.2j
    G = np.linalg.inv(z * np.eye(117) - H[:, None])
    ref = -np.trace(G, axis1=2, axis2=3).imag / np.pi
    assert rel(A.cpu().numpy(), ref.reshape(-1)) < TOL


def test_short_search_goes_without_the_forms():
    """One evaluation of N(mu) takes one solve, a longer search the Hessenberg forms; N agrees."""
    p, tau, om = _plan(3, 4)
    H, Sx, S = _inputs(2, len(om), 12, 5)
    a = dict(Sigx_k=dev(Sx), Sig_k_iw=dev(S))
    p.timing_enable(True)
    mu, n = p.chemical_potential(dev(H), 12.0, -0.5, 0.5, tol=1.0, **a)
    assert mu == 0.0 and "k_gj_inverse_smem" in p.timing_read() and "k_hessenberg" not in p.timing_read()
    mu2, n2 = p.chemical_potential(dev(H), n, -1e-9, 1e-9, tol=1e-10, **a)
    assert "k_hessenberg" in p.timing_read()
    assert abs(n2 - n) < 1e-7 and abs(mu2) < 1e-9


def test_failure_of_an_earlier_call_is_reported():
    """A Dyson step with an exactly singular matrix leaves its status; the search that follows
    reports it (as it does a zero pivot of its own), and the next one is clean."""
    from paper_1911_05633_gb300 import gw
    p, tau, om = _plan(1, 2)
    w = (2 * om + 1) * np.pi / 20.0
    S = np.zeros((2, len(om), 2, 2), np.complex128)
    S[:] = (1j * w)[None, :, None, None] * np.eye(2)
    p.dyson_green_tau(dev(np.zeros((2, 2, 2))), 0.0, Sig_k_iw=dev(S))
    H, Sx, S = _inputs(2, len(om), 2, 9)
    a = dict(Sigx_k=dev(Sx), Sig_k_iw=dev(S))
    with pytest.raises(gw.GwError) as e:
        p.chemical_potential(dev(H), 2.0, -4.0, 4.0, **a)
    assert e.value.status == 6
    p.chemical_potential(dev(H), 2.0, -4.0, 4.0, **a)
    p.sync()
