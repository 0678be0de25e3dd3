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


def _rows(plan, cell, kind, to_k, values):
    """Inputs of one transform, one slice per entry of `values`: a function of the slice's random
    numbers [.., elements]; flat, in the layout of the direction's input."""
    rng = np.random.default_rng(12)
    N, ns = plan.dense_n(kind), len(values)
    if to_k:
        out = np.zeros(plan.len(kind, ns), np.complex128)
        off = plan.offsets(kind)
        for e in range(len(off) - 1):
            n = int(off[e + 1] - off[e])
            for s, f in enumerate(values):
                out[ns * off[e] + s * n: ns * off[e] + (s + 1) * n] = f(rng.standard_normal(n) + 1j * rng.standard_normal(n))
        return out
    out = np.zeros((cell.n_k, ns, N * N), np.complex128)
    for s, f in enumerate(values):
        out[:, s] = f(rng.standard_normal((cell.n_k, N * N)) + 1j * rng.standard_normal((cell.n_k, N * N)))
    return out.reshape(-1)


def _slices(plan, cell, kind, to_k, x, ns):
    """The output of a transform as one array per slice."""
    N = plan.dense_n(kind)
    if to_k:
        return [y.reshape(-1) for y in x.reshape(cell.n_k, ns, N * N).transpose(1, 0, 2)]
    off = plan.offsets(kind)
    parts = [x[ns * off[e]: ns * off[e + 1]].reshape(ns, -1) for e in range(len(off) - 1)]
    return [np.concatenate([p[s] for p in parts]) for s in range(ns)]


SIZES = [1.0, 1e-280, 1e-291, 1e-295, 1e-300, 1e-305, 1e-308, 1e-318, 1e300, 1e305, 0.0]


@pytest.mark.parametrize("to_k", [False, True])
@pytest.mark.parametrize("same", [False, True])
def test_values_near_the_ends_of_the_range(to_k, same):
    """One size per slice, random over the mesh (or the classes) or one value that cancels in the
    sums.  Per slice: 2e-14 of its largest value as above, and half a unit of the subnormal numbers
    in each of the four products of a term, 64 terms: 128 x 2^-1074."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1911_05633_gb300 import gw
    cell = synth.mixed_species_cell(n_tau=9, n_orb=(4, 5), n_prod=(30, 35), kmesh=(3, 3, 3))
    a, b = gw.Plan.from_cell(cell), gw.Plan.from_cell(cell, fp64_products="fp64")

    def of(size):
        return lambda x: size * (np.full_like(x, -1.23) if same else x)

    F = dev(_rows(a, cell, "pb", to_k, [of(s) for s in SIZES]))
    run = (lambda p: p.fourier_R_to_k("pb", len(SIZES), F)) if to_k else (lambda p: p.fourier_k_to_R("pb", len(SIZES), F))
    a.timing_enable(True)
    got, ref = host(run(a)), host(run(b))
    a.sync()
    assert "k_lattice_tc" in a.timing_read()
    for size, x, y in zip(SIZES, *(_slices(a, cell, "pb", to_k, z, len(SIZES)) for z in (got, ref))):
        assert np.isfinite(y).all()
        tol = 2e-14 * size * (27 if to_k else 1) + 128 * 2.0 ** -1074
        assert max(np.abs(x.real - y.real).max(), np.abs(x.imag - y.imag).max()) <= tol, size


@pytest.mark.parametrize("to_k", [False, True])
def test_nan_and_infinities_pass_through(to_k):
    """One element of each kind among finite ones: the outputs that read it get what FP64
    arithmetic gives them, every other output its value (2e-14 as above, of sums of 27 terms)."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1911_05633_gb300 import gw
    cell = synth.mixed_species_cell(n_tau=9, n_orb=(4, 5), n_prod=(30, 35), kmesh=(3, 3, 3))
    a, b = gw.Plan.from_cell(cell), gw.Plan.from_cell(cell, fp64_products="fp64")
    x = _rows(a, cell, "pb", to_k, [lambda z: z] * 3)
    for i, bad in enumerate([np.nan, np.inf, -np.inf * 1j, complex(1.0, np.nan), complex(np.inf, np.inf)]):
        x[(2 * i + 1) * x.size // 11] = bad
    F = dev(x)
    run = (lambda p: p.fourier_R_to_k("pb", 3, F)) if to_k else (lambda p: p.fourier_k_to_R("pb", 3, F))
    a.timing_enable(True)
    got, ref = host(run(a)), host(run(b))
    a.sync()
    assert "k_lattice_tc" in a.timing_read()
    bad = ~np.isfinite(ref)
    assert 5 * 27 <= bad.sum() <= 5 * 27 * 3
    for g, r in ((got.real, ref.real), (got.imag, ref.imag)):
        assert np.array_equal(np.isnan(g), np.isnan(r)) and np.array_equal(g[np.isinf(r)], r[np.isinf(r)])
    assert np.abs(got[~bad] - ref[~bad]).max() <= 2e-14 * 27 * np.abs(x[np.isfinite(x)]).max()


def test_few_classes_on_a_small_mesh_stay_with_the_fp64_kernels():
    """One class per pair on three points, in blocks as wide as two warps: one step of the FP64
    kernels' warps per element; with every class kept, three."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1911_05633_gb300 import gw
    for cutoff, want in ((6.5, {"k_gather_k_to_R", "k_scatter_R_to_k"}), (0.0, {"k_lattice_tc"})):
        cell = synth.SynthCell("line", np.diag([30.0, 8.0, 8.0]), np.array([[i / 5, 0, 0] for i in range(5)]),
                               np.zeros(5, np.int32), [synth.Species("s", 3, 64, None)], (3, 1, 1), 20.0, 9, cutoff,
                               seed=5).build()
        p = gw.Plan.from_cell(cell)
        ns = 1 + 8_000_000 // (4 * cell.n_k * p.len("pb", 1))
        p.timing_enable(True)
        F = torch.ones(cell.n_k * ns * p.dense_n("pb") ** 2, dtype=torch.complex128, device="cuda")
        p.fourier_R_to_k("pb", ns, p.fourier_k_to_R("pb", ns, F))
        p.sync()
        assert set(p.timing_read()) == want


def test_status_of_an_earlier_call_stops_nothing():
    """A Dyson step with a singular matrix leaves its status for the next synchronisation; the
    transforms launched before that do their work."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1911_05633_gb300 import gw
    cell = synth.mixed_species_cell(n_tau=9, n_orb=(4, 5), n_prod=(30, 35), kmesh=(3, 3, 3))
    a, b = gw.Plan.from_cell(cell), gw.Plan.from_cell(cell, fp64_products="fp64")
    N, w = a.dense_n("orb"), (2 * cell.omega_idx + 1) * np.pi / cell.beta
    S = np.zeros((cell.n_k, len(w), N, N), np.complex128)
    S[:] = (1j * w)[None, :, None, None] * np.eye(N)  # i w - Sigma = 0
    a.dyson_green_tau(dev(np.zeros((cell.n_k, N, N))), 0.0, Sig_k_iw=dev(S))
    rng = np.random.default_rng(13)
    F = dev(rng.standard_normal(cell.n_k * 3 * a.dense_n("pb") ** 2))
    a.timing_enable(True)
    got = host(a.fourier_k_to_R("pb", 3, F))
    assert "k_lattice_tc" in a.timing_read()
    assert rel(got, host(b.fourier_k_to_R("pb", 3, F))) < 2e-14
    with pytest.raises(gw.GwError) as e:
        a.sync()
    assert e.value.status == 6
