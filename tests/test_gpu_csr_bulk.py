"""Rows of a sparse system in closed form (lb_csr_bulk.cu; needs an sm_103a
GPU) against the oracle, with its bars for sparse systems: the pattern exact,
values within 1e-12 of the larger of the entry and the summed magnitudes of its
terms; and against the join of Eq. (09), which takes over for more than four
channels: the same system with channels of rate zero added goes that way."""
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
    """(H or None, [(rate, L)]) as dense arrays."""
    r = np.random.default_rng(N + len(model))
    if model == "ladder":
        H, L, g = wl.ladder_model(N, 5)
        return H, [(g, L)]
    if model == "dimer":
        H, _, L, g, _ = wl.dimer_model(N)
        return H, [(g, L)]
    band = lambda k, c=1.0: np.diag((r.standard_normal(N - k) + 1j * r.standard_normal(N - k)) * c, k)  # noqa: E731
    if model == "complex":      # upper triangular, complex: the lower half cancels to rounding
        X = band(1)
        return X + X.conj().T + np.diag(r.standard_normal(N)), [(0.3, band(1))]
    if model == "two steps":    # next-nearest couplings, three channels, one with a diagonal
        X = band(2)
        return X + X.conj().T, [(0.2, band(1)), (1.1, np.ascontiguousarray(band(2).T)), (0.05, np.diag(r.standard_normal(N)).astype(complex))]
    if model == "graph":        # a random graph of degree about two: reordered pairs, common neighbours
        X, Y = np.zeros((N, N), complex), np.zeros((N, N), complex)
        X[r.integers(0, N, N), r.integers(0, N, N)] = r.standard_normal(N)
        Y[r.permutation(N), np.arange(N)] = r.standard_normal(N) + 1j * r.standard_normal(N)
        return X + X.conj().T, [(0.4, Y)]
    if model == "no H":
        return None, [(0.7, band(1))]
    if model == "weak channel":  # entries of the second far below the first's terms
        return None, [(1.0, band(1)), (1e-13, band(3))]
    if model == "weak edges":    # matrix elements over fifteen orders of magnitude
        L = band(1)
        L[np.arange(N - 1), np.arange(1, N)] *= 10.0 ** -r.integers(0, 16, N - 1)
        return None, [(1.0, L)]
    if model == "negative":
        return band(1) + band(1).conj().T, [(-0.2, band(1))]
    H, L, g = wl.ladder_model(N, 5)  # "hub": one level coupled to all
    L[0, :] = 0.3
    return H, [(g, L)]


@pytest.mark.parametrize("N", [64, 131])
@pytest.mark.parametrize("model", ["ladder", "dimer", "complex", "two steps", "graph", "no H", "weak channel",
                                   "weak edges", "negative", "hub"])
def test_closed_rows_equal_oracle_and_join(model, N):
    import paper_1912_01491_gb300 as lb
    with lb.Basis(N) as B, Oracle(N) as o:
        H, chans = _ops(model, N)
        h = None if H is None else B.expand(torch.tensor(H, device="cuda")).real.contiguous()
        ch, lps = [], []
        for g, L in chans:
            l = B.expand(torch.tensor(L, device="cuda"))
            nz = torch.nonzero(l.abs() > 0).flatten()
            ch.append((g, nz, l[nz].contiguous()))
            lps.append((nz.cpu().numpy(), l[nz].cpu().numpy()))
        zero = (0.0, ch[0][1][:1], ch[0][2][:1])
        a, b = lb.Csr(B, h=h, channels=ch), lb.Csr(B, h=h, channels=ch + [zero] * (5 - len(ch)))
        (rp, col, val, K), (rp2, col2, val2, _) = a.to_host(), b.to_host()
        assert np.array_equal(rp, rp2) and np.array_equal(col, col2)
        if model == "negative":  # the join keeps every entry it reaches there, the oracle does not
            assert np.abs(val - val2).max() <= 1e-12 * np.abs(val2).max()
            return
        orp, ocol, oval, oK, omag = lowrank_csr(o, None if h is None else h.cpu().numpy(), [g for g, _ in chans], lps,
                                                with_mag=True)
        assert np.array_equal(rp, orp) and np.array_equal(col, ocol)
        assert np.all(np.abs(val - oval) <= 1e-12 * np.maximum(np.abs(oval), np.abs(omag)))
        assert np.abs(K - oK).max() <= 1e-12 * max(np.abs(oK).max(), 1e-300) + 1e-18
        a.close()
        b.close()


@pytest.mark.parametrize("N", [70, 130])
def test_join_terms_and_repeated_entries(N):
    """The number of join terms does not depend on which rows are closed, and
    an index listed twice counts twice."""
    import paper_1912_01491_gb300 as lb
    with lb.Basis(N) as B:
        for model in ("ladder", "dimer", "graph"):
            H, [(g, L)] = _ops(model, N)
            l = B.expand(torch.tensor(L, device="cuda"))
            nz = torch.nonzero(l.abs() > 0).flatten()
            h = B.expand(torch.tensor(H, device="cuda")).real.contiguous()
            one = lb.Csr(B, h=h, channels=[(g, nz, l[nz].contiguous())])
            # a negative rate takes every row through the join: the same terms
            neg = lb.Csr(B, h=h, channels=[(-g, nz, l[nz].contiguous())])
            assert one.terms == neg.terms
            twice = lb.Csr(B, h=h, channels=[(g, torch.cat([nz, nz]), torch.cat([l[nz], l[nz]]) / 2)])
            for x, y in zip(one.to_host(), twice.to_host()):
                if x.dtype.kind == "f":
                    assert np.abs(x - y).max() <= 1e-13 * np.abs(x).max()
                else:
                    assert np.array_equal(x, y)
            for c in (one, neg, twice):
                c.close()
