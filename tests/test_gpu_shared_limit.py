"""The shared-memory limits that the dense assembly sets do not depend on the
call's N (needs an sm_103a GPU): a limit of the call's own size could be lowered
by another thread's smaller call between this call's setting and its launch."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_01491_gb300 import build
    build.build()


@pytest.mark.parametrize("algorithm,N,need", [("closed", 192, 8 * 32 * 513), ("join", 6, 16 * 10 * 512)])
def test_limit_covers_every_size(algorithm, N, need):
    """N = 192 is the first size whose closed form passes the default 48 KB;
    need: that of N = 512."""
    import paper_1912_01491_gb300 as lb
    with lb.Basis(N) as B:
        a = torch.zeros((B.M, B.M), dtype=torch.complex128, device="cuda")
        A = torch.empty((B.M, B.M), dtype=torch.float64, device="cuda")
        B.assemble_dense(a, A=A, algorithm=algorithm)
        torch.cuda.synchronize()
        assert not A.any()
        assert lb.native.load().lbi_dense_shared_limit(int(algorithm == "join")) >= need
        del a, A
    torch.cuda.empty_cache()
