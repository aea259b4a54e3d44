"""The closed assembly's overlapping kernels (lb_assemble.cu; needs a GPU): the
sizes where its block shapes change, against the join's kernels, which run one
after the other, and against its own kernels one after the other (the timed
entry point), whose bits it has to give; under graph capture likewise."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_01491_gb300 import build
    build.build()


def _inputs(N):
    M = N * N - 1
    gen = torch.Generator(device="cuda").manual_seed(N)
    l = torch.view_as_complex(torch.randn((M, 3, 2), generator=gen, device="cuda", dtype=torch.float64))
    return (l @ l.mH / M).contiguous(), torch.randn(M, generator=gen, device="cuda", dtype=torch.float64)


def _out(N):
    M = N * N - 1
    new = lambda *s: torch.full(s, float("nan"), device="cuda", dtype=torch.float64)  # noqa: E731
    return {"A": new(M, M), "Q": new(M, M), "R": new(M, M), "K": new(M)}


@pytest.mark.parametrize("N", [2, 3, 4, 5, 9, 16, 30, 31, 32, 33, 34, 64, 65])
def test_overlapped_equals_in_turn(N):
    import paper_1912_01491_gb300 as lb
    a, h = _inputs(N)
    with lb.Basis(N) as B:
        o, j = _out(N), _out(N)
        B.assemble_dense(a, h=h, **o, algorithm="closed")
        B.assemble_dense(a, h=h, **j, algorithm="join")
        # an entry is a sum of at most 16 N^2 terms f z a, |f|, |z| <= 2
        bound = 16 * N * N * 2.0 ** -52 * 4 * float(a.abs().max()) * 4
        for k in "ARK":
            assert float((o[k] - j[k]).abs().max()) <= bound + 2.0 ** -50 * float(o["Q"].abs().max()), k
        assert float((o["Q"] - j["Q"]).abs().max()) <= N * 2.0 ** -50 * float(h.abs().max())
        t = _out(N)
        B.assemble_dense_timed(a, h=h, A=t["A"], K=t["K"], algorithm="closed")
        for k in "AK":
            assert torch.equal(o[k], t[k]), k
        alone = torch.full_like(o["K"], float("nan"))
        B.assemble_dense(a, h=h, A=False, K=alone, algorithm="closed")
        assert float((alone - o["K"]).abs().max()) <= bound


@pytest.mark.parametrize("N", [7, 40])
def test_under_capture(N):
    import paper_1912_01491_gb300 as lb
    a, h = _inputs(N)
    with lb.Basis(N) as B:
        want, got = _out(N), _out(N)
        B.assemble_dense(a, h=h, **want, algorithm="closed")
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            B.assemble_dense(a, h=h, **got, algorithm="closed")
        for _ in range(2):
            for k in got:
                got[k].fill_(float("nan"))
            g.replay()
            torch.cuda.synchronize()
            for k in got:
                assert torch.equal(want[k], got[k]), k
