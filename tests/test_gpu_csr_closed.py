"""Rows of a sparse system in closed form (lb_csr_bulk.cu; needs an sm_103a
GPU) around the size from which they are taken, N = 128, and for one to four
channels: which rows the join still sums, and the result against the oracle with
its bars for sparse systems (pattern exact, values within 1e-12 of the larger of
the entry and the summed magnitudes of its terms)."""
import ctypes

import numpy as np
import pytest

import workloads as wl
from oracle import Oracle
from oracle.core import lowrank_csr

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_01491_gb300 import build
    build.build()


def _ops(model, N):
    r = np.random.default_rng(N + len(model))
    band = lambda k, c=1.0: np.diag((r.standard_normal(N - k) + 1j * r.standard_normal(N - k)) * c, k)  # noqa: E731
    if model == "ladder":
        H, L, g = wl.ladder_model(N, 5)
        return H, [(g, L)]
    if model == "dimer":
        H, _, L, g, _ = wl.dimer_model(N)
        return H, [(g, L)]
    X = band(1)
    H = X + X.conj().T
    ch = [(0.3, band(1)), (1.1, np.ascontiguousarray(band(1).T)), (0.05, np.diag(r.standard_normal(N)).astype(complex)),
          (0.2, band(2))]
    return H, ch[:int(model[0])] if model != "5 channels" else ch + [(0.1, band(1))]


@pytest.mark.parametrize("N,model", [(127, "ladder"), (128, "ladder"), (128, "dimer"), (128, "2 channels"),
                                     (128, "4 channels"), (128, "5 channels"), (160, "ladder"), (160, "dimer"),
                                     (160, "4 channels")])
def test_closed_rows_are_taken_and_equal_the_oracle(N, model):
    import paper_1912_01491_gb300 as lb
    joined = lb.native.load().lbi_csr_joined
    joined.restype, joined.argtypes = ctypes.c_longlong, [ctypes.c_void_p]
    with lb.Basis(N) as B, Oracle(N) as o:
        H, chans = _ops(model, N)
        h = B.expand(torch.tensor(H, device="cuda")).real.contiguous()
        ch, lps = [], []
        for g, L in chans:
            l = B.expand(torch.tensor(L, device="cuda"))
            nz = torch.nonzero(l.abs() > 0).flatten()
            ch.append((g, nz, l[nz].contiguous()))
            lps.append((nz.cpu().numpy(), l[nz].cpu().numpy()))
        c = lb.Csr(B, h=h, channels=ch)
        if N < 128 or model == "5 channels":
            assert joined(c._h) == c.M
        else:  # all but a few rows a level are far from the diagonal
            assert N - 1 <= joined(c._h) <= 40 * N
        rp, col, val, K = c.to_host()
        orp, ocol, oval, oK, omag = lowrank_csr(o, h.cpu().numpy(), [g for g, _ in chans], lps, with_mag=True)
        assert np.array_equal(rp, orp) and np.array_equal(col, ocol)
        assert np.all(np.abs(val - oval) <= 1e-12 * np.maximum(np.abs(oval), np.abs(omag)))
        assert np.abs(K - oK).max() <= 1e-12 * max(np.abs(oK).max(), 1e-300) + 1e-18
        c.close()
