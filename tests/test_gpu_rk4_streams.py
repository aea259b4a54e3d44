"""Dense RK4 of small systems (one cooperative launch each, lb_rk4_persist.cu)
on several streams at once, and beside other work (needs an sm_103a GPU)."""
import threading
import time

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_01491_gb300 import build
    build.build()


def _system(M, precision):
    import paper_1912_01491_gb300 as lb
    g = torch.Generator(device="cuda")
    g.manual_seed(M)
    A = torch.randn((M, M), generator=g, device="cuda", dtype=torch.float64) / M ** 0.5
    K = torch.randn(M, generator=g, device="cuda", dtype=torch.float64) / M
    if precision == "fp64":
        return A, None, None, K
    Ap, scale = (lb.pack_fp32(A), None) if precision == "fp32" else lb.pack_bf16(A)
    return Ap, scale, A, K


def _call(sys_, v, steps, precision, work, stream):
    import paper_1912_01491_gb300 as lb
    Ap, scale, A64, K = sys_
    lb.rk4_dense(Ap, K, v, 1e-3, steps, precision=precision, scale=scale, A64=A64,
                 correct_every=0 if precision == "fp64" else 7, work=work, stream=stream)


# a few rows a block, the edges of the rule on the warps of a block, a chip that one launch fills
@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("M", [99, 200, 201, 608, 609, 1216, 1217, 2432, 2433, 3400])
def test_several_integrations_at_once(M, precision):
    """Four streams from four threads, and products and an assembly on a fifth
    meanwhile: the bits of each integration alone."""
    import paper_1912_01491_gb300 as lb
    sys_, steps, n = _system(M, precision), 60, 4
    v0 = [torch.linspace(-1, 1 + i, M, dtype=torch.float64, device="cuda") for i in range(n)]
    works = [lb.rk4_workspace(M) for _ in range(n)]
    alone = [v.clone() for v in v0]
    for v in alone:
        _call(sys_, v, steps, precision, works[0], None)
    got = [v.clone() for v in v0]
    streams = [torch.cuda.Stream() for _ in range(n)]
    other = torch.cuda.Stream()
    X = torch.randn((1024, 1024), device="cuda")
    with lb.Basis(20) as B:
        a = torch.zeros((B.M, B.M), dtype=torch.complex128, device="cuda")
        out = torch.empty((B.M, B.M), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        ts = [threading.Thread(target=_call, args=(sys_, got[i], steps, precision, works[i], streams[i]))
              for i in range(n)]
        for t in ts:
            t.start()
        with torch.cuda.stream(other):
            for _ in range(10):
                X = X @ X / 1024
                B.assemble_dense(a, A=out, algorithm="closed", stream=other)
        for t in ts:
            t.join()
        torch.cuda.synchronize()
    for x, y in zip(got, alone):
        assert torch.equal(x, y) and torch.isfinite(x).all()


@pytest.mark.parametrize("N,precision", [(20, "fp32"), (30, "fp32"), (30, "bf16")])
def test_small_launches_share_the_chip(N, precision):
    """Eight integrations on eight streams take less than five and a half times
    as long as one (eight times if one launch keeps the others off every SM)."""
    import paper_1912_01491_gb300 as lb
    M, steps, n = N * N - 1, 3000, 8
    sys_ = _system(M, precision)
    v = [torch.zeros(M, dtype=torch.float64, device="cuda") for _ in range(n)]
    works = [lb.rk4_workspace(M) for _ in range(n)]
    streams = [torch.cuda.Stream() for _ in range(n)]

    def timed(k):
        best = 1e9
        for _ in range(4):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            for i in range(k):
                _call(sys_, v[i], steps, precision, works[i], streams[i])
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t0)
        return best

    assert timed(n) < 5.5 * timed(1)
