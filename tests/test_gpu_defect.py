"""The defect product (A64 - A_lp) v of the mixed-precision corrections, whose
differences are formed by integer operations (lb_rowsum.cuh; needs a GPU).

A_lp is A64 rounded to FP32 or to BF16 with row scales; A64 is then changed so
that every branch is taken: equal elements, zeros, opposite signs, other
binades, powers of two, subnormal and tiny elements.  A corrected step leaves
K + (A64 - A_lp) v in its workspace; with K = 0 that is compared
with exact rationals of the same inputs, the bound being the rounding of an
FP64 product of M terms.
"""
from fractions import Fraction

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


@pytest.mark.parametrize("M", [5, 128, 131, 700, 4099])
@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_defect_of_changed_elements(precision, M):
    import paper_1912_01491_gb300 as lb
    rng = np.random.default_rng(M)
    A = rng.standard_normal((M, M)) * 2.0 ** rng.integers(-6, 7, (M, M))
    A[rng.random((M, M)) < 0.1] = 0.0
    A64 = torch.tensor(A, device="cuda")
    scale = None
    if precision == "fp32":
        Ap = lb.pack_fp32(A64)
    else:
        Ap, scale = lb.pack_bf16(A64)
    odd = torch.tensor(rng.integers(0, 12, (M, M)), device="cuda")
    odd[:, M // 2:] = 99  # half of each row as packed
    A64 = torch.where(odd == 0, A64 * -1.0, A64)
    A64 = torch.where(odd == 1, A64 * 4.0, A64)
    A64 = torch.where(odd == 2, torch.full_like(A64, 0.5), A64)
    A64 = torch.where(odd == 3, A64 * 2.0 ** -600, A64)
    A64 = torch.where(odd == 4, torch.full_like(A64, 5e-324), A64)
    A64 = torch.where(odd == 5, A64 * (1 + 2.0 ** -52), A64).contiguous()
    v = torch.tensor(rng.standard_normal(M), device="cuda")
    K = torch.zeros(M, dtype=torch.float64, device="cuda")
    work = lb.rk4_workspace(M)
    lb.rk4_dense(Ap, K, v.clone(), 2.0 ** -30, 1, precision=precision, scale=scale, A64=A64, correct_every=1, work=work)
    at = 3 * ((8 * M + 255) // 256 * 256)  # behind the two stage vectors and the accumulator
    c = work[at:at + 8 * M].view(torch.float64).cpu().numpy()  # K plus the defect product
    low = Ap.double() if precision == "fp32" else Ap.view(torch.bfloat16).double() * scale.double()[:, None]
    D, vh = (A64 - low).cpu().numpy(), v.cpu().numpy()
    rows = np.arange(0, M, max(1, M // 16))
    want = np.array([float(sum(Fraction(float(d)) * Fraction(float(y)) for d, y in zip(D[i], vh))) for i in rows])
    # D is rounded once, the product M times
    assert np.all(np.abs(c[rows] - want) <= (M + 4) * 2.0 ** -53 * (np.abs(D[rows]) @ np.abs(vh)))
