"""Sparse assembly with negative rates (needs an sm_103a GPU): the join of
Eq. (09) then keeps every entry that it reaches, zeros included, and the rows in
closed form have no bound to decide by, so all rows have to come from the join.
The same system with channels of rate zero added takes the join alone."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_01491_gb300 import build
    build.build()


def _channel(B, rate, L):
    l = B.expand(torch.tensor(L, device="cuda"))
    nz = torch.nonzero(l.abs() > 0).flatten()
    return rate, nz, l[nz].contiguous()


# diagonal operators that are equal on many levels: rows whose entries all cancel, far from the diagonal too
@pytest.mark.parametrize("model", ["diagonal", "diagonal and H", "two channels"])
@pytest.mark.parametrize("N", [127, 128, 131])
def test_negative_rates_keep_the_pattern_of_the_join(N, model):
    import paper_1912_01491_gb300 as lb
    d = np.where(np.arange(N) < N // 2, 1.0, 0.3).astype(complex)
    up = np.diag(np.ones(N - 1), 1).astype(complex)
    with lb.Basis(N) as B:
        h = None
        ch = [_channel(B, -0.2, np.diag(d))]
        if model == "diagonal and H":
            h = B.expand(torch.tensor(np.diag(np.sin(np.arange(N) // 9)) + 0j, device="cuda")).real.contiguous()
        if model == "two channels":
            ch.append(_channel(B, 0.5, up))
        zero = (0.0, ch[0][1][:1], ch[0][2][:1])
        a, b = lb.Csr(B, h=h, channels=ch), lb.Csr(B, h=h, channels=ch + [zero] * (5 - len(ch)))
        (rp, col, val, K), (rp2, col2, val2, K2) = a.to_host(), b.to_host()
        assert np.array_equal(rp, rp2) and np.array_equal(col, col2)
        assert np.abs(val - val2).max() <= 1e-12 * np.abs(val2).max()
        assert np.abs(K - K2).max() <= 1e-12 * max(np.abs(K2).max(), 1e-300) + 1e-18
        a.close()
        b.close()
