"""The choice among equal forms: the in-place passes with the row width that the
rule picks (one row to the widest tile that fits, of boxes on both sides of the
form's limits) against the oracle, and sampled rows with lazy phases, which take
a width of their own.  Tolerances of the parity tests."""
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


# (n1, n2): rows of 2 n1 + 1, of which there are 2 n2 + 1
@pytest.mark.parametrize("dtype,tol", [("c64", 3e-5), ("c128", 3e-11)])
@pytest.mark.parametrize("n1,n2", [(3, 3), (4, 300), (60, 60), (200, 100), (288, 288), (320, 7), (700, 40), (1000, 3)])
def test_in_place_rows(P, monkeypatch, dtype, tol, n1, n2):
    monkeypatch.setenv("LSPLIT_NO_TILE", "1")
    p = W.bilayer_1d(n1, n2, 1.3, 0.9, ecut=1e9)
    x = W.random_state((p.M2, p.M1), 15)
    O.use_fft(True)
    try:
        for scheme in ("strang", "strang_stoch"):
            for no_ip in (("1", "0") if dtype == "c64" else ("0",)):
                monkeypatch.setenv("LSPLIT_NO_IP", no_ip)
                ctx = P.Context(p, dtype)
                psi = ctx.from_dense(x)
                ctx.step(psi, 3, 1e-3, scheme, seed=6)
                assert rel(ctx.to_dense(psi), O.step(p, x, 1e-3, scheme, 3, seed=6)) < tol, (scheme, no_ip)
    finally:
        O.use_fft(False)


@pytest.mark.parametrize("amp,scheme,n1,n2,tiles", [
    (1.0, "strang", 256, 256, True), (1.0, "strang", 320, 320, False), (1.0, "lie", 272, 272, True),
    (1.0, "lie", 288, 288, False), (6.0, "strang", 224, 224, True), (6.0, "strang", 272, 272, False),
    (6.0, "strang", 512, 128, False), (6.0, "lie", 224, 224, True), (6.0, "lie", 272, 272, False)])
def test_complex64_limit_of_the_tile_form(P, monkeypatch, amp, scheme, n1, n2, tiles):
    """Which complex64 boxes take the tile form (a pair of extent and factors
    that cannot be is refused where that form runs), and the same state either
    way at the limit."""
    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the limit counts tiles per SM")
    p = W.bilayer_1d(n1, n2, amp, 0.8 * amp, ecut=1e9)
    x = W.random_state((p.M2, p.M1), 16)
    ctx = P.Context(p, "c64")
    psi = ctx.from_dense(x)
    monkeypatch.setenv("LSPLIT_TILE", "5,1")
    if tiles:
        with pytest.raises(P.LsplitError):
            ctx.step(psi, 2, 1e-3, scheme)
    else:
        ctx.step(psi, 2, 1e-3, scheme)
    monkeypatch.delenv("LSPLIT_TILE")
    out = []
    for no_tile in ("0", "1"):
        monkeypatch.setenv("LSPLIT_NO_TILE", no_tile)
        ctx = P.Context(p, "c64")
        psi = ctx.from_dense(x)
        ctx.step(psi, 3, 1e-3, scheme)
        out.append(ctx.to_dense(psi))
    assert rel(out[0], out[1]) < 2e-6
