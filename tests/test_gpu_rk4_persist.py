"""RK4 of small dense systems in one cooperative launch (lb_rk4_persist.cu)
against the stage launches (needs an sm_103a GPU).

A captured call takes the stage launches, a direct one the cooperative launch;
both form the same sums in the same order, so the bar is equal bits.
"""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_01491_gb300 import build
    build.build()


def _system(M, spread, seed=1):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000 * M + seed)
    A = torch.randn((M, M), generator=g, device="cuda", dtype=torch.float64) / M ** 0.5
    if spread:  # entries over `spread` binades and a tenth of them zero: partial sums far apart
        A *= torch.exp2(-torch.randint(0, spread, (M, M), generator=g, device="cuda").double())
        A[torch.rand((M, M), generator=g, device="cuda") < 0.1] = 0.0
    K = torch.randn(M, generator=g, device="cuda", dtype=torch.float64) / M
    v = torch.randn(M, generator=g, device="cuda", dtype=torch.float64)
    return A, K, v


def _both(M, precision, correct, steps, snap_every=0, spread=0, offset=0):
    import paper_1912_01491_gb300 as lb
    A, K, v0 = _system(M, spread)
    scale = A64 = None
    Ap = A
    if precision != "fp64":
        A64 = A
        if precision == "fp32":
            Ap = lb.pack_fp32(A)
        else:
            Ap, scale = lb.pack_bf16(A)
    if offset:  # the matrix `offset` elements off its allocation's alignment
        raw = torch.empty(M * M + offset, dtype=Ap.dtype, device="cuda")
        raw[offset:].copy_(Ap.flatten())
        Ap = raw[offset:]
    kw = dict(precision=precision, scale=scale, A64=A64, correct_every=correct, snap_every=snap_every)
    v1, w1 = v0.clone(), lb.rk4_workspace(M)
    w1.fill_(255)  # stale words in the workspace
    n0 = lb.native.launch_count()
    s1 = lb.rk4_dense(Ap, K, v1, 1e-2, steps, work=w1, **kw)
    launched = lb.native.launch_count() - n0
    v2, w2 = v0.clone(), lb.rk4_workspace(M)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            s2 = lb.rk4_dense(Ap, K, v2, 1e-2, steps, work=w2, stream=torch.cuda.current_stream(), **kw)
        graph.replay()
    torch.cuda.synchronize()
    return launched, v0, v1, v2, s1, s2


# one element, a row shorter than a vector and than a warp, the edges of a chunk of 128, of two and of four rows a
# warp, rows beyond shared memory, the largest M of the range
@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("M", [1, 3, 31, 33, 99, 127, 128, 129, 257, 624, 899, 1680, 2432, 2499, 3400, 3600])
def test_one_launch_equals_stage_launches(M, precision):
    if precision == "fp32" and M > 3400:
        pytest.skip("beyond the range of the cooperative launch")
    launched, v0, v1, v2, _, _ = _both(M, precision, 0 if precision == "fp64" else 3, 7)
    assert launched == 1
    assert torch.isfinite(v1).all() and not torch.equal(v1, v0)
    assert torch.equal(v1, v2)


@pytest.mark.parametrize("precision,offset", [("fp64", 1), ("fp32", 1), ("fp32", 2), ("fp32", 3), ("bf16", 1),
                                              ("bf16", 3)])
@pytest.mark.parametrize("M", [99, 2000])
def test_any_alignment_of_the_matrix(M, precision, offset):
    _, _, v1, v2, _, _ = _both(M, precision, 0, 5, offset=offset)
    assert torch.equal(v1, v2)


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
@pytest.mark.parametrize("spread", [20, 60])
def test_partial_sums_far_apart(precision, spread):
    """Rows whose partial sums lie more than 30 binades apart take the FP64 additions."""
    _, _, v1, v2, _, _ = _both(255, precision, 2, 5, spread=spread)
    assert torch.equal(v1, v2)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("steps,every", [(1, 1), (6, 1), (7, 3), (2, 3)])
def test_snapshots(precision, steps, every):
    _, _, v1, v2, s1, s2 = _both(288, precision, 2 if precision == "fp32" else 0, steps, snap_every=every)
    assert torch.equal(v1, v2) and torch.equal(s1, s2)


def test_larger_systems_take_the_stage_launches():
    launched, _, v1, v2, _, _ = _both(3601, "fp64", 0, 2)
    assert launched == 8 and torch.equal(v1, v2)
