"""The dedicated passes of 16 x 16, 32 x 32 and 64 x 64 slices against the
oracle and against the general pass (LSPLIT_NO_FAST=1): both layers, last CTAs
that are not full, every mode, both types.

Tolerances: the parity tests' (1e-5 and 1e-11 for a step, three times that for
several); two FP32 transform forms of the same factor 3e-6, as the test of the
1D passes allows."""
import dataclasses

import numpy as np
import pytest

import oracle as O
import workloads as W
from tests._parity import rel

pytestmark = pytest.mark.gpu

TOL = {"c64": 1e-5, "c128": 1e-11}


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


def box(qa, qb):
    """Layer 1 with slices of extents qa, layer 2 with slices of extents qb."""
    p = W.twisted_2d(q=16, hmax=3, ecut=1e9)
    return dataclasses.replace(p, lo1=(-qa[0] // 2, 1 - qa[1]), q1=qa, lo2=(-3, -qb[1] // 2), q2=qb,
                               name=f"{qa}x{qb}")


# (number of slices of the other layer: 2, 6 and 256 among others, so that CTAs
# of 4 and 8 slices are cut off)
BOXES = [((16, 16), (2, 2)), ((2, 2), (16, 16)), ((16, 16), (16, 16)), ((32, 32), (4, 2)), ((2, 8), (32, 32)),
         ((32, 32), (16, 16)), ((64, 64), (2, 2)), ((2, 2), (64, 64))]


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("scheme", ["lie", "strang", "strang_kp", "yoshida4", "strang_stoch"])
def test_square_slices(P, monkeypatch, dtype, scheme):
    O.use_fft(True)
    try:
        for qa, qb in BOXES:
            p = box(qa, qb)
            x = W.random_state((p.M2, p.M1), 71)
            got = []
            for general in (False, True):
                if general:
                    monkeypatch.setenv("LSPLIT_NO_FAST", "1")
                else:
                    monkeypatch.delenv("LSPLIT_NO_FAST", raising=False)
                ctx = P.Context(p, dtype)
                psi = ctx.from_dense(x)
                ctx.step(psi, 3, 2e-3, scheme, seed=5, step0=1)
                assert float(psi[:, p.M1:].abs().sum()) == 0.0
                got.append(ctx.to_dense(psi))
            ref = O.step(p, x, 2e-3, scheme, 3, seed=5, step0=1)
            assert rel(got[0], ref) < 3 * TOL[dtype], (p.name, rel(got[0], ref))
            assert rel(got[0], got[1]) < (3e-6 if dtype == "c64" else 3e-12), (p.name, rel(got[0], got[1]))
    finally:
        O.use_fft(False)
