"""ls_density calls that follow one another or run at once on one context:
each gives what it gives alone."""
import threading

import numpy as np
import pytest

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


def state(P, ctx, p, seed):
    return ctx.from_dense(W.random_state((p.M2, p.M1), seed))


@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_larger_and_smaller_calls_in_turn(P, dtype):
    p = W.bilayer_1d(40, 70, 1.0, 0.8, ecut=1e9)
    ctx = P.Context(p, dtype)
    psi = state(P, ctx, p, 91)
    for npts in (5, 700, 64, 3000, 1):
        x = np.linspace(-1.3, 2.1, npts)
        assert np.array_equal(ctx.density(psi, x), P.Context(p, dtype).density(psi, x)), npts


@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_calls_of_several_threads(P, dtype):
    import torch
    p = W.bilayer_1d(100, 200, 1.0, 0.8, ecut=1e9)
    ctx = P.Context(p, dtype)
    jobs = [(state(P, ctx, p, 92 + i), np.linspace(-1.0 - i, 1.0, n), torch.cuda.Stream())
            for i, n in enumerate((40, 2500, 900, 300))]
    want = [ctx.density(psi, x) for psi, x, _ in jobs]
    torch.cuda.synchronize()
    bad = []

    def work(i):
        psi, x, st = jobs[i]
        for _ in range(30):
            if not np.array_equal(ctx.density(psi, x, stream=st), want[i]):
                bad.append(i)
    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert bad == []


@pytest.mark.parametrize("exp", [-70, 90, 110, 121])
def test_scaled_states(P, exp):
    """The sum is linear: a state times a power of two gives the value times it,
    up to the largest sums over m that complex64 holds (61 2^121; FP32 sums over
    m, 1e-5 as in the parity tests).  All coefficients 1: near x = 0 the sum
    over n adds up in one direction."""
    p = W.bilayer_1d(30, 200, 1.0, 0.8, ecut=1e9)
    ctx = P.Context(p, "c64")
    phi = np.ones((p.M2, p.M1), dtype=np.complex128)
    x = np.concatenate([[0.0], np.linspace(-1e-3, 1e-3, 70)])
    want = ctx.density(ctx.from_dense(phi), x)
    got = ctx.density(ctx.from_dense(phi * 2.0 ** exp), x) * 2.0 ** -exp
    assert np.abs(got - want).max() < 1e-5 * np.abs(want).max()
