"""Stochastic complex64 calls with long sampled factors (large taps): no further
from the FP64 oracle than the lazy phases (LSPLIT_NO_IP=1), whose kinetic phases
are exact.  The margin of 1.1 covers the scatter of rounding errors between the
two forms (over 4e3 elements and 20 steps their norms scatter by a few percent)."""
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


def error(got, ref):
    return np.linalg.norm(got - ref) / np.linalg.norm(ref)


# tau S / p max|v|, S / p = 8: the size of a sampled factor
@pytest.mark.parametrize("size", [0.01, 0.1, 0.14, 0.16, 0.3, 0.5, 0.7])
@pytest.mark.parametrize("scheme", ["lie_stoch", "strang_stoch"])
def test_no_further_off_than_lazy_phases(P, monkeypatch, scheme, size):
    p = W.bilayer_1d(64, 31, 1.0, 0.8, ecut=1e9)
    x = W.random_state((p.M2, p.M1), 51)
    O.use_fft(True)
    try:
        ref = O.step(p, x, size / 8, scheme, 20, seed=11, step0=2)
    finally:
        O.use_fft(False)
    err = {}
    for lazy in ("1", None):
        if lazy:
            monkeypatch.setenv("LSPLIT_NO_IP", lazy)
        else:
            monkeypatch.delenv("LSPLIT_NO_IP", raising=False)
        ctx = P.Context(p, "c64")
        psi = ctx.from_dense(x)
        ctx.step(psi, 20, size / 8, scheme, seed=11, step0=2)
        err[lazy] = error(ctx.to_dense(psi), ref)
    assert err[None] <= 1.1 * err["1"], err
    b = P.Batch([p, W.bilayer_1d(10, 12, 1.0, 0.8, ecut=1e9)], "c64")
    psi = b.empty()
    b.set_dense(psi, 0, x)
    b.step(psi, 20, size / 8, scheme, seed=11, step0=2)
    assert error(b.get_dense(psi, 0), ref) <= 1.1 * err["1"]
