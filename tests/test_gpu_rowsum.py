"""The combination of a row's FP32 partial sums in FP64 (lb_rowsum.cuh; needs
an sm_103a GPU)."""
import math

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_01491_gb300 import build
    build.build()


# the entries' spread in binades: within the fixed-point range, at its edge, beyond it (FP64 additions), and down to
# subnormal FP32 values
@pytest.mark.parametrize("gap", [0, 5, 29, 30, 31, 60, 130])
@pytest.mark.parametrize("precision", ["fp32", "bf16"])
@pytest.mark.parametrize("m", [1, 2, 65, 700, 1900])
def test_sum_of_partial_sums(m, precision, gap):
    """A = [[0, B], [0, 0]] and v = (0, 1): every stage has k = (B 1, 0), so a
    step of 6 gives (6 B 1, 1).  B holds signed powers of two in 120 columns,
    one to a partial sum, so the partial sums are exact and the result is the
    sum of the row's entries, off by at most one rounding of the sum (or, where
    FP64 additions form it, one of every addition) and three of the step."""
    import paper_1912_01491_gb300 as lb
    M = 2 * m
    g = torch.Generator().manual_seed(1000 * m + gap)
    n = min(m, 120)
    B = torch.exp2(torch.randint(-gap, 1, (m, n), generator=g).double())
    B *= 1.0 - 2.0 * torch.randint(0, 2, (m, n), generator=g).double()
    B[::3, ::2] = 0.0
    A = torch.zeros((M, M), dtype=torch.float64)
    A[:m, m:m + n] = B
    A = A.cuda()
    Ap, scale = (lb.pack_fp32(A), None) if precision == "fp32" else lb.pack_bf16(A)
    v = torch.cat([torch.zeros(m), torch.ones(m)]).double().cuda()
    lb.rk4_dense(Ap, torch.zeros(M, dtype=torch.float64, device="cuda"), v, 6.0, 1, precision=precision, scale=scale)
    v = v.cpu()
    assert torch.equal(v[m:], torch.ones(m, dtype=torch.float64))
    eps = 2.0 ** -53
    for s in range(m):
        row = B[s].tolist()
        want, size = 6.0 * math.fsum(row), math.fsum(abs(x) for x in row)
        bound = 4 * eps * abs(want) + (6 * 8 * eps * size if gap > 29 else 0.0)
        assert abs(v[s].item() - want) <= bound, (s, v[s].item(), want)


@pytest.mark.parametrize("M", [4257, 9001])
def test_stage_rows_in_rounds(M):
    """FP32 stages of more rows than an SM takes at once (one launch per stage,
    M = 4257 rows: one full round; 9001: three): one step against FP64 with the
    same FP32 matrix.  Each of the four stages adds at most (M + 4) 2^-24 of
    w = |A| |x| + |K| to its slope, x = v + dt k with |dt k| <= 2 dt w; factor 2
    to spare."""
    import paper_1912_01491_gb300 as lb
    gen = torch.Generator(device="cuda").manual_seed(M)
    A = (torch.randn((M, M), generator=gen, device="cuda") / M ** 0.5).contiguous()
    K = torch.randn(M, generator=gen, device="cuda", dtype=torch.float64) / M
    v0 = torch.randn(M, generator=gen, device="cuda", dtype=torch.float64)
    dt, A64, v = 1e-3, A.double(), v0.clone()
    lb.rk4_dense(A, K, v, dt, 1, precision="fp32", work=lb.rk4_workspace(M))
    k1 = A64 @ v0 + K
    k2 = A64 @ (v0 + 0.5 * dt * k1) + K
    k3 = A64 @ (v0 + 0.5 * dt * k2) + K
    k4 = A64 @ (v0 + dt * k3) + K
    ref = v0 + dt / 6 * (k1 + 2 * k2 + 2 * k3 + k4)
    w = A64.abs() @ v0.abs() + K.abs()
    bound = 2 * dt * (M + 4) * 2.0 ** -24 * (w + 2 * dt * (A64.abs() @ w)) + 2.0 ** -51 * v0.abs()
    assert bool(((v - ref).abs() <= bound).all())
