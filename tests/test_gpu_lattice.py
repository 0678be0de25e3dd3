"""Lattice transforms R <-> k on meshes with general phases (digit products on the tensor
cores) against the FP64 kernels of the same library, on random data: one and 32 mesh points'
neighbours, pairs with one class and with all, pairs without entries, one slice and several,
blocks of one element, reduced bases, two species.

Tolerance: both routes are sums of at most 64 products rounded like FP64, below 64 eps = 7e-15
of the largest terms; 2e-14 in the Frobenius norm.
"""
import numpy as np
import pytest

import synth
from test_gpu_parity import dev, host, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kmesh,cutoff,n_orb,n_prod,far,chained", [
    ((3, 1, 1), 0.0, (4, 5), (8, 19), None, True), ((3, 3, 3), 0.0, (4, 5), (8, 19), None, True),
    ((5, 2, 3), 6.0, (9, 9), (17, 16), None, True), ((3, 3, 3), 4.4, (1, 2), (1, 1), None, True),
    ((3, 2, 5), 7.2, (4, 5), (16, 33), 7, True), ((3, 1, 1), 6.5, "line", None, None, True),
    ((4, 4, 2), 0.0, (4, 5), (8, 19), None, False), ((3, 3, 4), 0.0, (4, 5), (8, 19), None, False)])
def test_against_fp64_kernels(kmesh, cutoff, n_orb, n_prod, far, chained):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1911_05633_gb300 import gw
    if n_orb == "line":  # five atoms in a row: pairs two apart have no entry, the ends meet in the next cell
        cell = synth.SynthCell("line", np.diag([30.0, 8.0, 8.0]), np.array([[i / 5, 0, 0] for i in range(5)]),
                               np.zeros(5, np.int32), [synth.Species("s", 3, 4, None)], kmesh, 20.0, 9, cutoff,
                               seed=5).build()
    else:
        cell = synth.mixed_species_cell(n_tau=9, n_orb=n_orb, n_prod=n_prod, kmesh=kmesh, cutoff=cutoff)
    if far:
        cell = synth.with_far_basis(cell, 4.4, [far] * 2, [min(n_prod)] * 2)
    a, b = gw.Plan.from_cell(cell), gw.Plan.from_cell(cell, fp64_products="fp64")
    rng = np.random.default_rng(11)
    z = lambda n: dev(rng.standard_normal(n) + 1j * rng.standard_normal(n))
    a.timing_enable(True)
    for kind in ("orb", "pb"):
        # many slices: the rule takes these kernels from a certain amount of work on
        for ns in (1, 3 + 40_000_000 // (4 * cell.n_k * a.len(kind, 1)) // (1 if kind == "orb" else 4)):
            F = z(cell.n_k * ns * a.dense_n(kind) ** 2)
            assert rel(host(a.fourier_k_to_R(kind, ns, F)), host(b.fourier_k_to_R(kind, ns, F))) < 2e-14
            R = z(a.len(kind, ns))
            assert rel(host(a.fourier_R_to_k(kind, ns, R)), host(b.fourier_R_to_k(kind, ns, R))) < 2e-14
            del F, R
    a.sync()
    b.sync()
    assert ("k_lattice_tc" in a.timing_read()) == chained
