"""Deterministic calls on two-dimensional tiles (several factors per pass):
against the oracle and against the in-place passes (LSPLIT_NO_TILE=1) at the
edges of the tiles, on boxes smaller than a halo, with taps of every class and
asymmetric potentials, over the FP64 range, and with two arrays in flight.

Tolerances: the forms differ by the rounding of the correction, at most a few
units of the last place per step (2e-6 and 1e-13 as the frames' own test and
FP64 rounding over 7 steps allow); the oracle's are those of the parity tests."""
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


def box(lo1, q1, lo2, q2, scale=0.7, harmonics=(1,), seed=3):
    """A 1D bilayer with complex (not even) potentials and a constant term."""
    rng = np.random.default_rng(seed)

    def pot():
        h, c = [[0]], [0.3 * scale]
        for k in harmonics:
            z = (rng.normal() + 1j * rng.normal()) * scale / 2
            h += [[k], [-k]]
            c += [z, np.conj(z)]
        return np.array(h, dtype=np.int64), np.array(c, dtype=np.complex128)
    (h1, c1), (h2, c2) = pot(), pot()
    return W.Problem(1, np.array([[2 * np.pi]]), np.array([[2 * np.pi / W.GOLDEN]]), (lo1,), (q1,), (lo2,), (q2,),
                     1e9, h1, c1, h2, c2, f"{q1}x{q2}")


def both(P, monkeypatch, p, x, dtype, n, tau, scheme):
    out = []
    for off in (False, True):
        if off:
            monkeypatch.setenv("LSPLIT_NO_TILE", "1")
        else:
            monkeypatch.delenv("LSPLIT_NO_TILE", raising=False)
        ctx = P.Context(p, dtype)
        psi = ctx.from_dense(x)
        ctx.step(psi, n, tau, scheme)
        assert float(psi[:, p.M1:].abs().sum()) == 0.0   # the pitch padding stays as it was
        out.append(ctx.to_dense(psi))
    return out


# result extents of a tile: 28 x 24, 24 x 24 (complex64), 10 x 10, 26 x 26,
# 58 x 58 and their halves (complex128); one less, equal and one more
BOXES = [(-3, 7, -4, 9), (-12, 24, -14, 28), (-12, 25, -14, 29), (-11, 23, -13, 27), (-5, 10, -26, 52),
         (-29, 58, -29, 59), (-32, 65, -100, 201), (0, 200, 5, 64), (-256, 513, -16, 33), (-9, 19, -350, 700)]


@pytest.mark.parametrize("dtype,tol,oracle_tol", [("c64", 2e-6, 1e-5), ("c128", 1e-13, 1e-11)])
@pytest.mark.parametrize("scheme,n", [("strang", 1), ("strang", 7), ("lie", 1), ("lie", 4), ("strang_kp", 3)])
def test_tile_form_matches_in_place_passes(P, monkeypatch, dtype, tol, oracle_tol, scheme, n):
    O.use_fft(True)
    try:
        for b in BOXES:
            p = box(*b)
            x = W.random_state((p.M2, p.M1), 31)
            tile, plain = both(P, monkeypatch, p, x, dtype, n, 1e-3, scheme)
            assert rel(tile, plain) < tol, (p.name, rel(tile, plain))
            ref = O.step(p, x, 1e-3, scheme, n)
            assert rel(tile, ref) < 3 * oracle_tol, (p.name, rel(tile, ref))
    finally:
        O.use_fft(False)


@pytest.mark.parametrize("dtype,tol", [("c64", 2e-6), ("c128", 1e-13)])
@pytest.mark.parametrize("scale,harmonics,tau", [(0.7, (1,), 1e-3), (3.0, (1,), 1e-3), (0.2, (1, 2), 1e-3),
                                                 (0.7, (1,), -1e-3), (0.0, (1,), 1e-3), (8.0, (1,), 4e-3)])
def test_tile_form_tap_classes(P, monkeypatch, dtype, tol, scale, harmonics, tau):
    """Narrow and wide taps, no taps at all, a backward step, and taps too
    large for the pairs of floats (the in-place form is taken: same state)."""
    p = box(-32, 65, -40, 81, scale, harmonics)
    x = W.random_state((p.M2, p.M1), 32)
    tile, plain = both(P, monkeypatch, p, x, dtype, 7, tau, "strang")
    assert rel(tile, plain) < tol, rel(tile, plain)


@pytest.mark.parametrize("dtype,mag", [("c64", 1e-30), ("c64", 1e30), ("c128", 1e-290), ("c128", 1e-40),
                                       ("c128", 1e40), ("c128", 1e290)])
def test_tile_form_range(P, dtype, mag):
    """The scheme is linear: a scaled state gives the scaled result (powers of
    two, so to rounding)."""
    p = box(-32, 65, -40, 81)
    s = 2.0 ** np.round(np.log2(mag))
    ctx = P.Context(p, dtype)
    x = W.random_state((p.M2, p.M1), 33)
    a, b = ctx.from_dense(x), ctx.from_dense(x * s)
    ctx.step(a, 3, 1e-3, "strang")
    ctx.step(b, 3, 1e-3, "strang")
    assert rel(ctx.to_dense(b) / s, ctx.to_dense(a)) < (1e-6 if dtype == "c64" else 1e-15)


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_tile_form_spreads_non_finite_values(P, dtype, bad):
    """A NaN or an infinity reaches the elements its factors reach and no others."""
    p = box(-32, 65, -40, 81)
    ctx = P.Context(p, dtype)
    x = W.random_state((p.M2, p.M1), 34)
    x[40, 30] = bad
    psi = ctx.from_dense(x)
    ctx.step(psi, 1, 1e-3, "lie")
    ok = np.isfinite(ctx.to_dense(psi))
    assert not ok[38:43, 28:33].any()
    ok[35:46, 25:36] = True
    assert ok.all()


@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_tile_form_two_arrays_on_two_streams(P, dtype):
    """Each array has its own second array: calls of one context on two
    streams at once give what they give one after the other."""
    import torch
    p = box(-128, 257, -128, 257)
    ctx = P.Context(p, dtype)
    xs = [ctx.from_dense(W.random_state((p.M2, p.M1), 35 + i)) for i in range(2)]
    want = [x.clone() for x in xs]
    for w in want:
        for _ in range(4):
            ctx.step(w, 6, 1e-3, "strang")
    streams = [torch.cuda.Stream() for _ in xs]
    torch.cuda.synchronize()
    for _ in range(4):
        for x, s in zip(xs, streams):
            ctx.step(x, 6, 1e-3, "strang", stream=s)
    torch.cuda.synchronize()
    for x, w in zip(xs, want):
        assert torch.equal(x, w)
