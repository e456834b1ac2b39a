"""Observables of 1D boxes in one pass (correlations with the potential's
harmonics instead of transforms) against FP64 NumPy on the same stored state.

Tolerance: sums of at most 1e5 terms accumulated in FP64 or in pairs of floats
with corrected low parts; 1e-13 of the sum of magnitudes leaves two orders for
the reference's own order of summation and transforms."""
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


def box(lo1, q1, lo2, q2, harmonics):
    rng = np.random.default_rng(6)

    def pot():
        h, c = [[0]], [0.4]
        for k in harmonics:   # one-sided and complex: Re(.) makes the potential real
            h.append([k])
            c.append(rng.normal() + 1j * rng.normal())
        return np.array(h, dtype=np.int64), np.array(c, dtype=np.complex128)
    (h1, c1), (h2, c2) = pot(), pot()
    return W.Problem(1, np.array([[2 * np.pi]]), np.array([[2 * np.pi / W.GOLDEN]]), (lo1,), (q1,), (lo2,), (q2,),
                     1e9, h1, c1, h2, c2, f"{q1}x{q2}")


# boxes below, at and above a warp item of 512; harmonics beyond the box length,
# at half of an even one, negative, and more than the one pass takes
CASES = [((-32, 65, -40, 81), (1,)), ((-3, 7, -4, 9), (1, 2, 30)), ((0, 8, 0, 16), (4, 8, -3)), ((5, 1, -2, 5), (1,)),
         ((-256, 512, -3, 7), (2, -2)), ((-256, 513, 9, 33), (1, -5)), ((-100, 1100, -5, 64), tuple(range(1, 9))),
         ((-30, 61, -20, 41), tuple(range(1, 12)))]


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("mag", [1.0, 1e-25, 1e22])
def test_observables_1d(P, dtype, mag):
    ct = np.complex64 if dtype == "c64" else np.complex128
    for b, hs in CASES:
        p = box(*b, hs)
        x = (W.random_state((p.M2, p.M1), 41) * mag).astype(ct)
        x[: p.M2 // 3] *= 1e-12          # rows far below the others
        x[p.M2 // 2] = 0
        chi = (W.random_state((p.M2, p.M1), 42) * mag).astype(ct)
        ctx = P.Context(p, dtype)
        o = ctx.observables(ctx.from_dense(x), ctx.from_dense(chi))
        x, chi = x.astype(np.complex128), chi.astype(np.complex128)
        k = O.wavevectors(p)[..., 0]
        a2 = np.abs(x) ** 2
        n = a2.sum()
        v1, v2 = (O.grid_potential(h, c, q) for h, c, q in ((p.v1_h, p.v1_c, p.q1), (p.v2_h, p.v2_c, p.q2)))
        y1, y2 = np.fft.ifft(x, axis=1, norm="ortho"), np.fft.ifft(x, axis=0, norm="ortho")
        want = {"norm": (n, n), "ekin": ((0.5 * k * k * a2).sum(),) * 2,
                "epot1": ((np.abs(y1) ** 2 * v1[None, :]).sum(), n * np.abs(v1).max()),
                "epot2": ((np.abs(y2) ** 2 * v2[:, None]).sum(), n * np.abs(v2).max())}
        # more harmonics than the one pass takes: FP32 transforms for complex64
        tol = 1e-13 if len(hs) <= 8 or dtype == "c128" else 1e-6
        for key, (ref, scale) in want.items():
            assert abs(o[key] - ref) <= (tol if key.startswith("epot") else 1e-13) * scale, (p.name, hs, key)
        assert abs(o["kmean"][0] - (k * a2).sum()) <= 1e-13 * (np.abs(k) * a2).sum()
        assert abs(o["overlap"] - np.vdot(chi, x)) <= 1e-13 * np.linalg.norm(chi) * np.linalg.norm(x)


def test_observables_1d_non_finite(P):
    p = box(-32, 65, -40, 81, (1,))
    ctx = P.Context(p, "c64")
    for bad in (np.nan, np.inf):
        x = W.random_state((p.M2, p.M1), 43)
        x[7, 9] = bad
        o = ctx.observables(ctx.from_dense(x))
        assert not np.isfinite(o["norm"]) and not np.isfinite(o["energy"])
