"""The places of the rows of the structure lists (lb_basis.cu; needs an
sm_103a GPU): whole lists against the oracle where a row passes a warp's 32
triples, and the invariants of the lists at larger N."""
import numpy as np
import pytest

from oracle import Oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_01491_gb300 import build
    build.build()


@pytest.mark.parametrize("N", [13, 17, 18, 33, 34, 40])
def test_lists_equal_the_oracles(N):
    import paper_1912_01491_gb300 as lb
    with lb.Basis(N) as B, Oracle(N) as o:
        for w in "fd":
            idx, val = B.structure(w)
            oi, ov = o.structure(w)
            assert B.structure_count(w) == len(ov)
            assert np.array_equal(idx.cpu().numpy(), oi)
            assert np.abs(val.cpu().numpy() - ov).max() < 1e-14


@pytest.mark.parametrize("N", [64, 65, 129, 256, 300])
def test_lists_are_sorted_and_complete(N):
    """Strictly ascending (m, n, s) with m <= n <= s, and the sums that the
    normalization of the basis fixes: sum_ns f_mns^2 = 2N and sum_ns d_mns^2 =
    2 (N^2 - 4)/N for every m."""
    import paper_1912_01491_gb300 as lb
    M = N * N - 1
    with lb.Basis(N) as B:
        for w, want in (("f", 2.0 * N), ("d", 2.0 * (N * N - 4.0) / N)):
            idx, val = B.structure(w)
            i = idx.to(torch.int64)
            assert bool((i[:, 0] <= i[:, 1]).all()) and bool((i[:, 1] <= i[:, 2]).all())
            assert bool((i[:, 0] >= 0).all()) and bool((i[:, 2] < M).all())
            key = (i[:, 0] * M + i[:, 1]) * M + i[:, 2]
            assert bool((key[1:] > key[:-1]).all())
            # each unordered triple stands for all its distinct orders
            sums = torch.zeros(M, dtype=torch.float64, device="cuda")
            v2 = val * val
            mn, ns = i[:, 0] == i[:, 1], i[:, 1] == i[:, 2]
            distinct = ~mn & ~ns
            for c in range(3):  # (n, s) ordered pairs beside element c
                mult = torch.where(distinct, 2.0, 0.0)
                if c == 2:
                    mult = torch.where(mn & ~ns, 1.0, mult)  # (m, m | s)
                if c == 0:
                    mult = torch.where(mn & ~ns, 2.0, mult)  # (m | m, s), (m | s, m)
                    mult = torch.where(ns & ~mn, 1.0, mult)
                    mult = torch.where(mn & ns, 1.0, mult)
                if c == 1:
                    mult = torch.where(ns & ~mn, 2.0, mult)
                sums.index_add_(0, i[:, c], v2 * mult)
            assert (sums - want).abs().max().item() < 1e-11 * want
