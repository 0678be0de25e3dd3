"""The FP64 P and Sigma over symmetric pairs (chained digit products) against the FP64-only
kernels of the same library, on random G, W~ and v without any symmetry, at the sizes where
tiles end: one function, one pair, 16 and 17 product functions, 64 (the largest), 55 pairs
(n = 10), an odd node count, two species, reduced bases; and at sizes outside its limits.

Both routes round like FP64 sums of at most n^2 K = 6400 terms: relative errors of each are
below sqrt(6400) 2^-52 < 2e-14, and two of them differ by less than 1e-13 in the Frobenius norm.
"""
import numpy as np
import pytest

import synth
from test_gpu_parity import dev, host, rel

pytestmark = pytest.mark.gpu


def _cell(n_orb, n_prod, n_tau, far=None):
    cell = synth.mixed_species_cell(n_tau=n_tau, n_orb=n_orb, n_prod=n_prod, kmesh=(2, 1, 1))
    if far:
        cell = synth.with_far_basis(cell, 4.4, [far] * 2, [min(n_prod)] * 2)
    return cell


@pytest.mark.parametrize("n_orb,n_prod,n_tau,far,chained", [
    ((4, 1), (25, 1), 9, None, True), ((5, 3), (16, 17), 10, None, True), ((5, 9), (33, 48), 11, None, True),
    ((9, 4), (64, 8), 10, None, True), ((10, 9), (32, 30), 9, None, True), ((10, 9), (49, 30), 9, None, False), ((9, 9), (48, 48), 12, 20, True),
    ((11, 4), (20, 8), 9, None, False), ((9, 9), (65, 20), 9, None, False), ((4, 4), (24, 8), 9, None, False),
    ((9, 9), (11, 8), 9, None, False)])
def test_pairs_against_fp64_kernels(n_orb, n_prod, n_tau, far, chained):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1911_05633_gb300 import gw
    cell = _cell(n_orb, n_prod, n_tau, far)
    a, b = gw.Plan.from_cell(cell), gw.Plan.from_cell(cell, fp64_products="fp64")
    rng = np.random.default_rng(7)
    z = lambda n: dev((rng.standard_normal(n) + 1j * rng.standard_normal(n)) * 10.0 ** rng.uniform(-6, 3, n))
    G, W, v = z(a.len("orb", n_tau)), z(a.len("pb", n_tau)), z(a.len("pb", 1))
    a.timing_enable(True)
    P = host(a.polarizability_tau(G))
    S, X = a.self_energy_tau(G, W, v_R=v)
    a.sync()
    a.timing_enable(False)
    assert ("k_chain" in a.timing_read()) == chained
    S2, X2 = b.self_energy_tau(G, W, v_R=v)
    assert rel(P, host(b.polarizability_tau(G))) < 1e-13
    assert rel(host(S), host(S2)) < 1e-13
    assert rel(host(X), host(X2)) < 1e-13
    b.sync()


def _plans(n_tau):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1911_05633_gb300 import gw
    cell = _cell((5, 9), (33, 48), n_tau)
    a, b = gw.Plan.from_cell(cell), gw.Plan.from_cell(cell, fp64_products="fp64")
    a.timing_enable(True)
    return cell, a, b


def _slices(p, kind, n, x):
    """A flat buffer in the entry layout as views [slice][elements] per entry."""
    off = p.offsets(kind)
    return [x[n * off[e]: n * off[e + 1]].reshape(n, -1) for e in range(len(off) - 1)]


def _agree(plan, kind, n, got, ref, floor):
    """Per node: 1e-13 in the Frobenius norm (as above) beside `floor` per element."""
    for i in range(n):
        g, r = (np.concatenate([q[i] for q in _slices(plan, kind, n, x)]) for x in (got, ref))
        size = max(np.abs(r).max(), 2.0 ** -1022)  # the squares stay in the range
        assert np.isfinite(r).all()
        assert np.linalg.norm((g - r) / size) <= 1e-13 * np.linalg.norm(r / size) + np.sqrt(r.size) * floor / size, i


def test_values_near_the_ends_of_the_range():
    """P, Sigma and Sigma_x of inputs of one size per node against the FP64-only kernels.  The
    digits take subnormal elements of M, W~ and v for zero: less than 2^-1022 each, in a sum with
    the coefficients of both atoms (and G for Sigma)."""
    sizes = [1.0, 1e-140, 1e-145, 1e-148, 1e-152, 1e-160, 1e150]
    nt = 2 * len(sizes) - 1
    cell, a, b = _plans(nt)
    rng = np.random.default_rng(8)
    z = lambda n: rng.standard_normal(n) + 1j * rng.standard_normal(n)
    G, W, G1 = z(a.len("orb", nt)), z(a.len("pb", nt)), z(a.len("orb", nt))
    node = np.array(sizes + sizes[-2::-1])  # G(tau) and G(beta - tau) of one size
    for x, kind, sc in ((G, "orb", node), (W, "pb", node ** 2)):
        for y in _slices(a, kind, nt, x):
            y *= sc[:, None]
    c_k = max(np.abs(s.C).sum(axis=(1, 2)).max() for s in cell.species)  # sum over (L, L'') of |C[K][L][L'']|
    c = max(np.abs(s.C).sum() for s in cell.species)
    _agree(a, "pb", nt, host(a.polarizability_tau(dev(G))), host(b.polarizability_tau(dev(G))), 8 * c_k ** 2 * 2.0 ** -1022)
    for size in (1.0, 1e-300, 1e300):
        v = dev(z(a.len("pb", 1)) * size)
        S, X = a.self_energy_tau(dev(G1), dev(W), v_R=v)
        S2, X2 = b.self_energy_tau(dev(G1), dev(W), v_R=v)
        for n, got, ref in ((nt, S, S2), (1, X, X2)):
            _agree(a, "orb", n, host(got), host(ref), 4 * c ** 2 * np.abs(G1).max() * 2.0 ** -1022)
    a.sync()
    t = a.timing_read()
    assert {"k_chain", "k_slice_w_units", "k_sigma_pairs"} <= set(t) and "k_self_energy_fp64" not in t


def test_nan_and_infinities_pass_through():
    """One element that is no number in G, W~ and v: the outputs that take it are no numbers, as in
    FP64 arithmetic, the others keep their values (1e-13 as above)."""
    nt = 9
    cell, a, b = _plans(nt)
    rng = np.random.default_rng(9)
    z = lambda n: rng.standard_normal(n) + 1j * rng.standard_normal(n)
    G, W, v, G1 = z(a.len("orb", nt)), z(a.len("pb", nt)), z(a.len("pb", 1)), z(a.len("orb", nt))
    bad = [np.nan, np.inf, complex(1.0, np.nan), complex(2.0, -np.inf)]
    for x in (G, W, v):
        x[[(2 * i + 1) * x.size // 9 for i in range(4)]] = bad
    S, X = a.self_energy_tau(dev(G1), dev(W), v_R=dev(v))
    S2, X2 = b.self_energy_tau(dev(G1), dev(W), v_R=dev(v))
    pairs = [(S, S2), (X, X2), (a.polarizability_tau(dev(G)), b.polarizability_tau(dev(G)))]
    a.sync()
    assert "k_chain" in a.timing_read()
    for got, ref in ((host(x), host(y)) for x, y in pairs):
        ok = np.isfinite(ref)
        assert np.array_equal(np.isfinite(got), ok) and 0 < ok.sum() < ok.size
        assert rel(got[ok], ref[ok]) < 1e-13
