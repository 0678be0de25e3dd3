"""The tau <-> i omega transforms on the tensor cores at both ends of the FP64 range, with NaN and
with infinities, against the FP64 kernel of the same library: one size per element over its
whole row of nodes or frequencies.

Tolerance per size: both are sums of K <= 64 products with coefficients up to t, good to a few
2^-52 of K t size: 1e-13 K t size; and the digits take subnormal inputs for zero, 2^-1022 each.
"""
import numpy as np
import pytest

import synth
from test_gpu_parity import dev, host

pytestmark = pytest.mark.gpu

SIZES = [1.0, 1e-280, 1e-292, 1e-297, 1e-303, 1e-307, 1e-315, 1e300, 0.0]
FORMS = [("F", "tau_to_iw", "orb", "general"), ("F", "iw_to_tau", "orb", "general"), ("B", "tau_to_iw", "pb", "general"),
         ("B", "iw_to_tau", "pb", "general"), ("B", "tau_to_iw", "pb", "mirror"), ("B", "tau_to_iw", "pb", "mirror_nonneg"),
         ("B", "iw_to_tau", "pb", "real")]


def _case(stat, direction, kind, structure, n_tau):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1911_05633_gb300 import gw
    cell = synth.mixed_species_cell(n_tau=n_tau, n_orb=(4, 5), n_prod=(8, 19), kmesh=(2, 1, 1))
    a, b = gw.Plan.from_cell(cell), gw.Plan.from_cell(cell, fp64_products="fp64")
    T = np.abs(a.transform_matrix(stat, direction))
    n_out, n_in = T.shape
    off = a.offsets(kind)
    rng = np.random.default_rng(21)
    z = rng.standard_normal((n_in, off[-1])) + 1j * rng.standard_normal((n_in, off[-1]))
    if structure.startswith("mirror"):
        z = 0.5 * (z + z[::-1].conj())
    if structure == "real":
        z = z.real.astype(np.complex128)

    def run(p, x):  # x [slice][element] -> [slice][element]
        flat = np.concatenate([x[:, off[e]:off[e + 1]].reshape(-1) for e in range(len(off) - 1)])
        out = host(p.transform_tau_iw(stat, direction, kind, dev(flat), out=dev(np.zeros(n_out * off[-1])), structure=structure))
        p.sync()
        return np.concatenate([out[n_out * off[e]: n_out * off[e + 1]].reshape(n_out, -1) for e in range(len(off) - 1)], 1)
    a.timing_enable(True)
    return a, b, T, z, run


@pytest.mark.parametrize("n_tau", [12, 33])
@pytest.mark.parametrize("form", FORMS)
def test_values_near_the_ends_of_the_range(form, n_tau):
    a, b, T, z, run = _case(*form, n_tau)
    size = np.array([SIZES[i % len(SIZES)] for i in range(z.shape[1])])
    x = z * size
    got, ref = run(a, x), run(b, x)
    assert "k_oz_transform" in a.timing_read() and np.isfinite(ref).all()
    tol = 2 * T.shape[1] * T.max() * (4e-13 * size + 4 * 2.0 ** -1022)
    assert (np.abs(got.real - ref.real) <= tol).all() and (np.abs(got.imag - ref.imag) <= tol).all()


@pytest.mark.parametrize("form", FORMS)
def test_nan_and_infinities_pass_through(form):
    a, b, T, z, run = _case(*form, 12)
    nt = z.shape[0]
    for i, bad in enumerate([np.nan, np.inf, -np.inf]):
        z[2, 5 + 7 * i] = bad
        if form[3].startswith("mirror"):
            z[nt - 3, 5 + 7 * i] = bad
    got, ref = run(a, z), run(b, z)
    assert "k_oz_transform" in a.timing_read()
    ok = np.isfinite(ref)
    assert np.array_equal(np.isfinite(got), ok) and 0 < (~ok).sum() <= 3 * T.shape[0]
    assert np.abs(got[ok] - ref[ok]).max() <= 1e-12 * T.shape[1] * T.max()
