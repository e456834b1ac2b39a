"""Calls so long that the factors' scalar parts Lambda of the interaction frame
decay far: one call against the same call cut into short ones.

Tolerance: both round every factor; added up coherently over F factors that is
at most F 2^-24 (complex64) and F 2^-53 (complex128) on each side."""
import numpy as np
import pytest

import workloads as W
from tests._parity import rel

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


# |Lambda| of the whole call: 1e-13 and 1e-19 (complex64), 0.27 (complex128)
@pytest.mark.parametrize("dtype,amp,tau,scheme,n,cuts", [
    ("c64", 200.0, 1e-3, "strang", 2000, 100),
    ("c64", 200.0, 1e-3, "lie", 2003, 100),
    ("c64", 200.0, 1e-3, "strang_kp", 2000, 100),
    ("c64", 50.0, 1e-3, "strang", 50000, 50),
    ("c128", 3.4, 1e-3, "lie", 230000, 4),
])
@pytest.mark.parametrize("tiles", [True, False])
def test_long_call_equals_its_pieces(P, monkeypatch, dtype, amp, tau, scheme, n, cuts, tiles):
    if not tiles:
        if dtype == "c128" or n > 10000:
            pytest.skip("the in-place passes of complex128 are not in the frame; one long case is enough")
        monkeypatch.setenv("LSPLIT_NO_TILE", "1")
    p = W.bilayer_1d(13, 9, amp, 0.8 * amp, ecut=1e9)
    ctx = P.Context(p, dtype)
    x = W.random_state((p.M2, p.M1), 71)
    one, cut = ctx.from_dense(x), ctx.from_dense(x)
    ctx.step(one, n, tau, scheme)
    for k in range(cuts):
        ctx.step(cut, n // cuts + (n % cuts if k == 0 else 0), tau, scheme)
    tol = 2 * 3 * n * (2.0 ** -24 if dtype == "c64" else 2.0 ** -53)
    assert rel(ctx.to_dense(one), ctx.to_dense(cut)) < tol


@pytest.mark.parametrize("scheme", ["strang", "lie"])
def test_long_batched_call_equals_its_pieces(P, scheme):
    probs = [W.bilayer_1d(13, 9, 200.0, 150.0, ecut=1e9), W.bilayer_1d(40, 20, 3.0, 2.0, ecut=1e9)]
    b = P.Batch(probs, "c64")
    xs = [W.random_state((p.M2, p.M1), 80 + i) for i, p in enumerate(probs)]
    one, cut = b.empty(), b.empty()
    for i, x in enumerate(xs):
        b.set_dense(one, i, x)
        b.set_dense(cut, i, x)
    b.step(one, 2003, 1e-3, scheme)
    for k in range(100):
        b.step(cut, 20 + (3 if k == 0 else 0), 1e-3, scheme)
    for i in range(2):
        assert rel(b.get_dense(one, i), b.get_dense(cut, i)) < 2 * 3 * 2003 * 2.0 ** -24


@pytest.mark.parametrize("tiles", [True, False])
@pytest.mark.parametrize("amp", [1.0, 2.4, 3.4])
def test_long_complex128_call_keeps_the_norm(P, monkeypatch, tiles, amp):
    """20000 Strang steps are unitary: the norm may move by the random roundings
    of 60000 factors (60000^(1/2) 2^-53 = 3e-14) and by the factors' tables
    (1e-18 each, 6e-14 if it all adds up); four times their sum."""
    if not tiles:
        monkeypatch.setenv("LSPLIT_NO_TILE", "1")
    p = W.bilayer_1d(16, 12, amp, 0.8 * amp, ecut=1e9)
    ctx = P.Context(p, "c128")
    x = W.random_state((p.M2, p.M1), 72)
    psi = ctx.from_dense(x)
    ctx.step(psi, 20000, 1e-3, "strang")
    got, want = np.linalg.norm(ctx.to_dense(psi)), np.linalg.norm(x)
    assert abs(got / want - 1) < 4e-13


@pytest.mark.parametrize("scheme", ["strang_stoch", "lie_stoch"])
def test_long_stochastic_batch_in_pieces(P, scheme):
    """Beyond one graph of launches a stochastic batched call is replayed in
    pieces: same samples and states as the call cut anywhere, and device memory
    that does not grow with the steps (64 MB: the graph of 60000 steps in one
    piece holds 120000 or more launches)."""
    import torch
    probs = [W.bilayer_1d(9, 6, 2.0, 1.5, ecut=1e9), W.bilayer_1d(5, 12, 1.0, 0.7, ecut=1e9)]
    b = P.Batch(probs, "c64")
    xs = [W.random_state((p.M2, p.M1), 85 + i) for i, p in enumerate(probs)]
    one, cut = b.empty(), b.empty()
    for i, x in enumerate(xs):
        b.set_dense(one, i, x)
        b.set_dense(cut, i, x)
    n = 3503
    b.step(one, n, 1e-3, scheme, seed=4, step0=7)
    b.step(cut, 1203, 1e-3, scheme, seed=4, step0=7)
    b.step(cut, n - 1203, 1e-3, scheme, seed=4, step0=7 + 1203)
    for i in range(2):
        assert rel(b.get_dense(one, i), b.get_dense(cut, i)) < 2 * 3 * n * 2.0 ** -24
    free = torch.cuda.mem_get_info()[0]
    b.step(one, 60000, 1e-3, scheme, seed=4)
    assert free - torch.cuda.mem_get_info()[0] < 64 << 20


def test_pieces_with_a_full_list_of_graphs(P):
    """The graph of a call's rest is the oldest of the batch's cached ones when
    the graph of its pieces is built: it must not be the one that makes room."""
    probs = [W.bilayer_1d(9, 6, 2.0, 1.5, ecut=1e9)]
    b = P.Batch(probs, "c64")
    x = W.random_state((probs[0].M2, probs[0].M1), 88)
    psi, want = b.empty(), b.empty()
    b.set_dense(psi, 0, x)
    b.set_dense(want, 0, x)
    steps = [11, 1, 2, 3, 1011]          # four cached graphs, the rest of 1011 = 1000 + 11 the oldest
    step0 = 0
    for n in steps:
        b.step(psi, n, 1e-3, "strang_stoch", seed=5, step0=step0)
        step0 += n
    b2 = P.Batch(probs, "c64")
    b2.step(want, 500, 1e-3, "strang_stoch", seed=5)
    b2.step(want, step0 - 500, 1e-3, "strang_stoch", seed=5, step0=500)
    assert rel(b.get_dense(psi, 0), b2.get_dense(want, 0)) < 2 * 3 * step0 * 2.0 ** -24
