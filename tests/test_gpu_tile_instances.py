"""Every instance of the tile kernels (half-width of the taps, extent, factors
per pass; LSPLIT_TILE fixes the last two, which a rule on the box's size picks
otherwise) against the oracle and the in-place passes: tiles of one and of
several rows and columns, ragged ends, seams on both axes, boxes smaller than a
tile with its halo.  Tolerances of the tile form's own tests."""
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


TAU = 1e-3
# amplitudes of the first and second harmonic for which the taps of a factor of
# duration TAU have the given half-width
AMPS = {("c64", 2): (0.3, 0.0), ("c64", 3): (6.0, 0.0),
        ("c128", 3): (0.6, 0.0), ("c128", 4): (2.6, 0.0), ("c128", 5): (0.12, 0.03)}


def box(lo1, q1, lo2, q2, amps):
    h = np.array([[0], [1], [-1], [2], [-2]], dtype=np.int64)
    z1, z2 = amps[0] / 2 * np.exp(0.7j), amps[1] / 2 * np.exp(-0.4j)
    c = np.array([0.2, z1, np.conj(z1), z2, np.conj(z2)], dtype=np.complex128)
    return W.Problem(1, np.array([[2 * np.pi]]), np.array([[2 * np.pi / W.GOLDEN]]), (lo1,), (q1,), (lo2,), (q2,),
                     1e9, h, c, h, c, f"{q1}x{q2}")


def half_width(amps, dtype, s, q=129):
    """The class of the taps of exp(-i s v) - 1: dropped l1 tail below 2^-30 or
    2^-48, and 5 narrowed to 4 where that still holds; the kernels start at 2
    and 3; complex128 needs taps of at most 2^-7 in all and 2^-30 beyond 2."""
    x = np.arange(q) / q
    v = 0.2 + amps[0] * np.cos(2 * np.pi * x + 0.7) + amps[1] * np.cos(4 * np.pi * x - 0.4)
    c = np.fft.fft(np.exp(-1j * s * v) - 1) / q
    t = np.array([np.abs(c[d]) + np.abs(c[-d]) for d in range(1, q // 2)])   # t[d - 1]
    eps = 2.0 ** (-30 if dtype == "c64" else -48)
    B = next(b for b in (2, 3, 5, 8) if t[b:].sum() <= eps)
    if B == 5 and dtype == "c128" and t[4:].sum() <= eps:
        B = 4
    if dtype == "c128":
        assert t.sum() < 2.0 ** -7 and np.abs(c[3:-2]).max() < 2.0 ** -30
    return max(B, 2 if dtype == "c64" else 3)


CASES = [("c64", b, 32, nf) for b in (2, 3) for nf in (1, 2, 3)]
CASES += [("c128", b, e, nf) for b in (3, 4, 5) for e in (16, 32, 64) for nf in (1, 2, 3) if (b, e) != (5, 16)]
BOXES = [(-3, 11, -4, 13), (-32, 65, -100, 201), (0, 200, 5, 64), (-64, 129, -20, 41), (-29, 58, -61, 124)]


@pytest.mark.parametrize("dtype,bv,ext,nf", CASES)
def test_instance(P, monkeypatch, dtype, bv, ext, nf):
    amps = AMPS[dtype, bv]
    assert half_width(amps, dtype, TAU) == bv
    tol, oracle_tol = (2e-6, 3e-5) if dtype == "c64" else (1e-13, 3e-11)
    O.use_fft(True)
    try:
        for k, b in enumerate(BOXES):
            p = box(*b, amps)
            x = W.random_state((p.M2, p.M1), 36)
            for scheme, n in (("strang", 6), ("lie", 3 + k), ("strang_kp", 4)):
                out = {}
                for tile in (f"{ext},{nf}", None):
                    if tile:
                        monkeypatch.setenv("LSPLIT_TILE", tile)
                        monkeypatch.delenv("LSPLIT_NO_TILE", raising=False)
                    else:
                        monkeypatch.setenv("LSPLIT_NO_TILE", "1")
                    ctx = P.Context(p, dtype)
                    psi = ctx.from_dense(x)
                    try:
                        ctx.step(psi, n, TAU, scheme)
                    except P.LsplitError:
                        # two factors of one layer leave no result
                        assert tile and nf > 1 and ext <= 4 * bv
                        break
                    assert float(psi[:, p.M1:].abs().sum()) == 0.0
                    out[tile] = ctx.to_dense(psi)
                if len(out) < 2:
                    continue
                assert rel(out[f"{ext},{nf}"], out[None]) < tol, (p.name, scheme)
                ref = O.step(p, x, TAU, scheme, n)
                assert rel(out[f"{ext},{nf}"], ref) < oracle_tol, (p.name, scheme)
    finally:
        O.use_fft(False)


@pytest.mark.parametrize("shape", [(401, 401), (513, 513), (129, 2049)])
@pytest.mark.parametrize("amps", [(0.6, 0.0), (2.6, 0.0), (0.12, 0.03)])
def test_large_boxes_as_the_rule_picks(P, monkeypatch, shape, amps):
    """Boxes on which the rule takes 64 x 64 tiles and several factors per pass."""
    p = box(-(shape[0] // 2), shape[0], -(shape[1] // 2), shape[1], amps)
    x = W.random_state((p.M2, p.M1), 37)
    for n in (1, 4, 7):
        monkeypatch.delenv("LSPLIT_NO_TILE", raising=False)
        ctx = P.Context(p, "c128")
        psi = ctx.from_dense(x)
        ctx.step(psi, n, TAU, "strang")
        monkeypatch.setenv("LSPLIT_NO_TILE", "1")
        ctx = P.Context(p, "c128")
        plain = ctx.from_dense(x)
        ctx.step(plain, n, TAU, "strang")
        assert rel(ctx.to_dense(psi), ctx.to_dense(plain)) < 1e-13, (p.name, n)
    O.use_fft(True)
    try:
        assert rel(ctx.to_dense(psi), O.step(p, x, TAU, "strang", 7)) < 3e-11
    finally:
        O.use_fft(False)
