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
