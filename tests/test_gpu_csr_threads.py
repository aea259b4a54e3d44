"""First integrations of one sparse system from several threads at once
(needs an sm_103a GPU): its layout is made once, under a lock."""
import threading

import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_01491_gb300 import build
    build.build()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("N", [12, 60])
def test_threads_make_one_layout(N, precision):
    import paper_1912_01491_gb300 as lb
    r = np.random.default_rng(N)
    H, L, g = wl.ladder_model(N, 3)
    with lb.Basis(N) as B:
        l = B.expand(torch.tensor(L, device="cuda")).cpu().numpy()
        ch = [(g, np.flatnonzero(np.abs(l) > 0), l[np.abs(l) > 0])]
        v0 = r.standard_normal(B.M)
        for _ in range(5):
            s = lb.System(B, H=H, channels=ch, format="csr")
            out, start = [None] * 6, threading.Barrier(6)

            def work(i):
                start.wait()
                out[i] = s.integrate(v0, 0.03, 1e-3, precision=precision, correct_every=0 if precision == "fp64" else 5)

            ts = [threading.Thread(target=work, args=(i,)) for i in range(6)]
            for t in ts:
                t.start()
            for t in ts:
                t.join()
            again = s.integrate(v0, 0.03, 1e-3, precision=precision, correct_every=0 if precision == "fp64" else 5)
            assert np.isfinite(again).all() and all(np.array_equal(o, again) for o in out)
            s.close()
