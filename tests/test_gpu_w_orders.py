"""The W solve for orders N_PB that are no multiple of 128 (the tensor-core inverse beside an
identity) against the FP64 Gauss-Jordan solve of the same plan inputs: one below the first
order it takes, the first, odd ones on both sides of a tile, the largest; and inputs it hands
to the FP64 inverse: a v(q) too ill-conditioned for the FP32 start, and scales outside FP32.
A reversed identity for v(q) makes every column of the FP32 start change rows.

Tolerance: both solves are FP64-accurate, kappa(v) eps N < 1e3 1e-16 4e2 = 4e-11 < 1e-10.  For
the ill-conditioned v both are FP64 eliminations with error kappa eps sqrt(N) = 1e7 1.1e-16 14
= 1.6e-8 of W each, so 1e-6 of the larger W~ is a wide bound; without the FP64 inverse the
FP32 start is off by order one there.
"""
import numpy as np
import pytest

import synth
from test_gpu_parity import TOL, dev, host, rel

pytestmark = pytest.mark.gpu


def _plans(n_prod, **kw):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1911_05633_gb300 import gw
    if n_prod == "8 atoms":
        cell = synth.make_config(1, kmesh=(2, 1, 1), n_tau=12)  # N_PB 384
    else:
        cell = synth.mixed_species_cell(n_tau=10, n_orb=(4, 5), n_prod=n_prod, kmesh=(2, 2, 1))
    G = dev(cell.green_k_tau())
    a, b = gw.Plan.from_cell(cell, **kw), gw.Plan.from_cell(cell, w_solver="gauss_jordan", **kw)
    P = a.transform_tau_iw("B", "tau_to_iw", "pb", a.polarizability_tau(a.green_k_to_R(G)))
    return cell, a, b, P


@pytest.mark.parametrize("n_prod,sym", [((43, 44), True), ((44, 44), True), ((63, 64), True), ((65, 64), True),
                                        ((100, 101), True), ((128, 127), False), ((128, 128), True)])
def test_orders(n_prod, sym):
    cell, a, b, P = _plans(n_prod, no_symmetry=not sym)
    v = dev(cell.coulomb()[0])
    W = host(a.screened_W_iw(P, v))
    a.sync()
    ref = host(b.screened_W_iw(P, v))
    b.sync()
    assert rel(W, ref) < TOL


@pytest.mark.parametrize("low,scale,bound", [(1e-7, 1.0, 1e-6), (0.5, 1e-60, TOL), (0.5, 1e60, TOL)])
def test_left_to_the_fp64_inverse(low, scale, bound):
    cell, a, b, P = _plans((100, 101))
    rng = np.random.default_rng(3)
    N = cell.n_pb_total
    Q = np.linalg.qr(rng.standard_normal((N, N)))[0]
    v = (Q * np.geomspace(low, 1.0, N)) @ Q.T
    vq = dev(np.broadcast_to(scale * 0.5 * (v + v.T), (cell.n_k, N, N)))
    P = P * (1e-3 / scale)
    W = host(a.screened_W_iw(P, vq))
    a.sync()
    ref = host(b.screened_W_iw(P, vq))
    b.sync()
    assert np.isfinite(W).all() and rel(W, ref) < bound


@pytest.mark.parametrize("n_prod", [(64, 64), (100, 101), (128, 128), "8 atoms"])
def test_every_pivot_off_the_diagonal(n_prod):
    cell, a, b, P = _plans(n_prod)
    rng = np.random.default_rng(4)
    N = cell.n_pb_total
    v = np.eye(N)[::-1] + (lambda x: x + x.T)(0.02 / np.sqrt(N) * rng.standard_normal((N, N)))
    vq = dev(np.broadcast_to(v, (cell.n_k, N, N)))
    P = P * (0.1 / P.abs().max().item())  # v^-1 - P: a reversed identity and a small rest
    W = host(a.screened_W_iw(P, vq))
    a.sync()
    ref = host(b.screened_W_iw(P, vq))
    b.sync()
    assert rel(W, ref) < TOL


def test_route():
    """The tensor-core inverse from order 88 on, while one frequency's matrices fit the caller's cap."""
    for n_prod, kw, tensor in (((43, 44), {}, False), ((44, 44), {}, True), ((44, 44), {"workspace_bytes": 1 << 20}, False),
                               ((128, 127), {}, True), ((128, 127), {"workspace_bytes": 8 << 20}, False)):
        cell, a, b, P = _plans(n_prod, **kw)
        a.timing_enable(True)
        a.screened_W_iw(P, dev(cell.coulomb()[0]))
        a.sync()
        assert ("k_gj_inverse_f32" in a.timing_read()) == tensor, (n_prod, kw)


@pytest.mark.parametrize("n_prod", [(43, 44), (44, 44), (100, 101), (128, 128)])
def test_singular_v_is_reported_as_such(n_prod):
    """A v(q) with a zero row: status 6, as by the FP64 elimination, not a wait that gave up; and
    the plan works again after it."""
    from paper_1911_05633_gb300 import gw
    cell, a, b, P = _plans(n_prod)
    N = cell.n_pb_total
    v = cell.coulomb()[0].reshape(cell.n_k, N, N).copy()
    ref = host(b.screened_W_iw(P, dev(v)))
    bad = v.copy()
    bad[1, 7] = bad[1, :, 7] = 0.0
    for p in (a, b):
        p.screened_W_iw(P, dev(bad))
        with pytest.raises(gw.GwError) as e:
            p.sync()
        assert e.value.status == 6
    W = host(a.screened_W_iw(P, dev(v)))
    a.sync()
    assert rel(W, ref) < TOL
