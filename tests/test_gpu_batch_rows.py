"""Row distribution of the batched RK4 kernels (lb_batch.cu; needs a GPU): the
lanes per row change at M = 32, 96 and 256, a warp takes one to four rows at a
time, and a block holds as many rows as fit and streams the rest.  A row's sum
does not depend on any of it, so the bits are the same at every cluster size,
and each trajectory stays within a rounding bound of FP64 numpy RK4: over a
step of size dt the four stages each add M + 8 roundings of magnitude at most
w = |A| |v| + |K|, with a factor 2 to spare; storage and products in FP32
count 2^-24 each (M + 4 of them)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

NS = [2, 3, 5, 6, 10, 11, 16, 17, 26, 33, 40, 47, 64]


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_01491_gb300 import build
    build.build()


def _numpy_rk4(A, K, v, dt, steps):
    f = lambda x: A @ x + K  # noqa: E731
    for _ in range(steps):
        k1 = f(v)
        k2 = f(v + 0.5 * dt * k1)
        k3 = f(v + 0.5 * dt * k2)
        k4 = f(v + dt * k3)
        v = v + dt / 6 * (k1 + 2 * k2 + 2 * k3 + k4)
    return v


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_same_bits_at_every_cluster_size(precision):
    import paper_1912_01491_gb300 as lb
    gen = torch.Generator(device="cuda").manual_seed(5)
    steps, dt = 3, 1e-3
    b = lb.Batch(NS)
    M = [n * n - 1 for n in NS]
    v0 = [torch.randn(m, generator=gen, device="cuda", dtype=torch.float64) for m in M]
    v = [x.clone() for x in v0]
    for r, m in enumerate(M):
        g = torch.randn((m, 8, 2), generator=gen, device="cuda", dtype=torch.float64)
        l = torch.view_as_complex(g)
        b.set(r, (l @ l.mH / m).contiguous(), torch.randn(m, generator=gen, device="cuda", dtype=torch.float64), v[r])
    b.assemble("closed")
    b.set_precision(precision)
    first = None
    for C in (1, 2, 4, 8, 16):
        for r in range(len(NS)):
            b.set_cluster(r, C)
            v[r].copy_(v0[r])
        b.integrate(dt, steps, correct_every=2 if precision == "fp32" else 0)
        out = [x.clone() for x in v]
        if first is None:
            first = out
        for r in range(len(NS)):
            assert torch.equal(out[r], first[r]), (C, NS[r])
    u, per = (2.0 ** -24, 4) if precision == "fp32" else (2.0 ** -53, 8)
    for r, m in enumerate(M):
        A, K = b.system(r)
        x0 = v0[r].cpu().numpy()
        ref = _numpy_rk4(A, K, x0, dt, steps)
        w = np.abs(A) @ np.abs(x0) + np.abs(K)
        bound = 2 * 4 * steps * dt * (m + per) * u * w.max() + 4 * steps * 2.0 ** -53 * np.abs(ref).max()
        assert np.abs(first[r].cpu().numpy() - ref).max() <= bound, NS[r]
    b.close()
