"""Two contexts on two threads building graphs of the tile form at once: the
kernels' shared-memory limits belong to the process, so one thread's smaller
pass must not lower the limit under the other's larger one."""
import threading

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


def test_two_contexts_on_two_threads(P):
    import torch
    p = W.bilayer_1d(256, 220, 1.0, 0.8, ecut=1e9)
    x = W.random_state((p.M2, p.M1), 61)
    ctxs = [P.Context(p, "c128") for _ in range(2)]
    psis = [c.from_dense(x) for c in ctxs]
    errors = []

    def work(i):
        st = torch.cuda.Stream()
        try:
            for n in range(1, 60):
                ctxs[i].step(psis[i], n, 1e-3, "lie" if n & 1 else "strang", stream=st)
        except Exception as e:   # a refused launch
            errors.append(e)
        st.synchronize()
    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert errors == []
    assert torch.equal(psis[0], psis[1])
