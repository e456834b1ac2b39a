"""Observables of 1D boxes where FP32 products or their moments would leave the
float range: large states on long rows (the second moment grows as m^2 |psi|^2),
and overlaps with a state so small, or so far apart, that only FP64 keeps the
products.  Tolerance as for the other magnitudes: 1e-13 of the sum of magnitudes."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2103_14897_gb300 import build as B
    B.build()
    import paper_2103_14897_gb300 as P
    P.load_library()
    return P


def check(P, p, x, chi):
    ctx = P.Context(p, "c64")
    o = ctx.observables(ctx.from_dense(x), ctx.from_dense(chi))
    x, chi = x.astype(np.complex128), chi.astype(np.complex128)
    k = O.wavevectors(p)[..., 0]
    a2 = np.abs(x) ** 2
    assert abs(o["norm"] - a2.sum()) <= 1e-13 * a2.sum()
    assert abs(o["ekin"] - (0.5 * k * k * a2).sum()) <= 1e-13 * (0.5 * k * k * a2).sum()
    assert abs(o["kmean"][0] - (k * a2).sum()) <= 1e-13 * (np.abs(k) * a2).sum()
    assert abs(o["overlap"] - np.vdot(chi, x)) <= 1e-13 * np.abs(chi * x).sum()


@pytest.mark.parametrize("mag", [1e9, 1e11, 1e13, 1e15, 1e17, 1e18, 1e-11, 1e-13])
def test_large_and_small_states_on_long_rows(P, mag):
    for n1, n2 in [(256, 8), (1024, 5)]:
        p = W.bilayer_1d(n1, n2, 1.0, 0.8, ecut=1e9)
        x, chi = ((W.random_state((p.M2, p.M1), s) * mag * np.sqrt(p.M1 * p.M2)).astype(np.complex64) for s in (1, 2))
        check(P, p, x, chi)


@pytest.mark.parametrize("psi_mag,chi_mag", [(1.0, 1e-35), (1e-10, 1e-30), (1e-30, 1e-12), (1e8, 1e-36), (1e10, 1e17)])
def test_small_overlaps(P, psi_mag, chi_mag):
    p = W.bilayer_1d(256, 8, 1.0, 0.8, ecut=1e9)
    x = (W.random_state((p.M2, p.M1), 3) * psi_mag * np.sqrt(p.M1 * p.M2)).astype(np.complex64)
    chi = (W.random_state((p.M2, p.M1), 4) * chi_mag * np.sqrt(p.M1 * p.M2)).astype(np.complex64)
    check(P, p, x, chi)


def test_overlap_of_states_that_hardly_meet(P):
    """Each is large where the other is tiny, within every row."""
    p = W.bilayer_1d(256, 8, 1.0, 0.8, ecut=1e9)
    left = np.where(np.arange(p.M1) < p.M1 // 2, 1.0, 1e-36)
    x = (W.random_state((p.M2, p.M1), 5) * left).astype(np.complex64)
    chi = (W.random_state((p.M2, p.M1), 6) * left[::-1]).astype(np.complex64)
    check(P, p, x, chi)
