"""Stochastic complex64 calls in the interaction frame (sampled slices get
their factors, K(T) once at the end) against the oracle and against the lazy
phases (LSPLIT_NO_IP=1), and the parallel sampler against the oracle's.

Tolerances: the parity tests' (1e-5 for a step, three times that for several);
the two forms differ by rounding only (2e-6, as the frames' own test)."""
import numpy as np
import pytest

import oracle as O
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


def with_offset(p, v0):
    """A constant term in both potentials: the factors' scalar parts are phases."""
    return p.with_potentials(np.append(p.v1_c, v0), np.append(p.v2_c, v0), np.append(p.v1_h, [[0]], axis=0),
                             np.append(p.v2_h, [[0]], axis=0))


@pytest.mark.parametrize("scheme", ["lie_stoch", "strang_stoch"])
@pytest.mark.parametrize("frac_den", [1, 3, 8])
def test_single_context(P, monkeypatch, scheme, frac_den):
    O.use_fft(True)
    try:
        for n1, n2 in [(3, 4), (16, 40), (40, 16), (512, 5), (5, 600)]:
            p = with_offset(W.bilayer_1d(n1, n2, 1.3, 0.9, ecut=1e9), 0.4)
            x = W.random_state((p.M2, p.M1), 51)
            got = {}
            for lazy in ("1", None):
                if lazy:
                    monkeypatch.setenv("LSPLIT_NO_IP", lazy)
                else:
                    monkeypatch.delenv("LSPLIT_NO_IP", raising=False)
                ctx = P.Context(p, "c64", frac_den=frac_den)
                psi = ctx.from_dense(x)
                ctx.step(psi, 5, 1e-3, scheme, seed=11, step0=2)
                got[lazy] = ctx.to_dense(psi)
            assert rel(got[None], got["1"]) < 2e-6, (p.M1, p.M2)
            if frac_den == 8:
                ref = O.step(p, x, 1e-3, scheme, 5, seed=11, step0=2)
                assert rel(got[None], ref) < 3e-5, (p.M1, p.M2)
    finally:
        O.use_fft(False)


@pytest.mark.parametrize("scheme", ["lie_stoch", "strang_stoch"])
def test_batch(P, scheme):
    """Instances with several rows per CTA, one row per CTA, and wide taps."""
    probs = [with_offset(q, 0.3) for q in W.batch_1d(count=6, seed=9, nmin=3, nmax=30)]
    probs += [W.bilayer_1d(400, 300, 1.1, 0.6, ecut=1e9), W.bilayer_1d(30, 20, 9.0, 8.0, ecut=1e9)]
    b = P.Batch(probs, "c64")
    psi = b.empty()
    xs = [W.random_state((p.M2, p.M1), 60 + i) for i, p in enumerate(probs)]
    for i, x in enumerate(xs):
        b.set_dense(psi, i, x)
    b.step(psi, 4, 2e-3, scheme, seed=3, step0=1)
    O.use_fft(True)
    try:
        for i, p in enumerate(probs):
            ref = O.step(p, xs[i], 2e-3, scheme, 4, seed=3 + i, step0=1)
            assert rel(b.get_dense(psi, i), ref) < 3e-5, (i, p.name)
    finally:
        O.use_fft(False)


@pytest.mark.parametrize("n", [0, 3, 15, 127, 128, 1024, 2048])
def test_sampler(P, n):
    for frac_den in (1, 3, 8):
        p = W.bilayer_1d(n, 5, 1.0, 0.8, ecut=1e9)
        ctx = P.Context(p, "c64", frac_den=frac_den)
        S = p.M1
        k = max(1, S // frac_den)
        got = ctx.samples(2, seed=77, g0=5, count=3)
        for r in range(3):
            assert np.array_equal(got[r], np.asarray(O.sample_slices(S, k, 77, 5 + r))), (S, frac_den, r)


def test_batch_timeout_hook(P):
    """The hook that makes a wait unsatisfiable still ends a stochastic call
    with LS_ERR_TIMEOUT, and the batch works again afterwards."""
    probs = W.batch_1d(count=3, seed=2, nmin=8, nmax=20)
    b = P.Batch(probs, "c64")
    psi = b.empty()
    b.debug(True, 0.2)
    with pytest.raises(P.LsplitError) as e:
        b.step(psi, 2, 1e-3, "strang_stoch", seed=1)
    assert e.value.code == P.LS_ERR_TIMEOUT
    b.debug(False, 1.0)
    xs = [W.random_state((p.M2, p.M1), 90 + i) for i, p in enumerate(probs)]
    for i, x in enumerate(xs):
        b.set_dense(psi, i, x)
    b.step(psi, 2, 1e-3, "strang_stoch", seed=1)
    for i, p in enumerate(probs):
        assert rel(b.get_dense(psi, i), O.step(p, xs[i], 1e-3, "strang_stoch", 2, seed=1 + i)) < 3e-5
