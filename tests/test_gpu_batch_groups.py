"""Groups of the batched RK4 (lb_batch.cu; needs an sm_103a GPU): streamed rows
on both sides of the length from which they are asked for ahead, FP64 slices that
share an SM, and the order in which the groups of different cluster sizes go."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_01491_gb300 import build
    build.build()


def _batch(Ns, precision, seed=3):
    import paper_1912_01491_gb300 as lb
    gen = torch.Generator(device="cuda").manual_seed(seed)
    b = lb.Batch(Ns)
    v, keep = [], {}
    for r, N in enumerate(Ns):
        M = N * N - 1
        if N not in keep:
            l = torch.view_as_complex(torch.randn((M, 8, 2), generator=gen, device="cuda", dtype=torch.float64))
            keep[N] = ((l @ l.mH / M).contiguous(), torch.randn(M, generator=gen, device="cuda", dtype=torch.float64))
        v.append(torch.randn(M, generator=gen, device="cuda", dtype=torch.float64))
        b.set(r, *keep[N], v[r])
    b.assemble()
    b.set_precision(precision)
    return b, v


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_mixed_groups_give_the_bits_of_one_at_a_time(precision):
    """M = 1848, 1935 (the line lies at 1900), 2024 and small ones, every cluster
    size in one call, against each realization in a batch of its own."""
    Ns = [44, 43, 45, 44, 43, 5, 9, 16, 30, 36]
    Cs = [16, 8, 4, 2, 1, 2, 1, 4, 8, 16]
    b, v = _batch(Ns, precision)
    v0 = [x.clone() for x in v]
    for r, C in enumerate(Cs):
        b.set_cluster(r, C)
    corr = 2 if precision == "fp32" else 0
    b.integrate(1e-3, 5, correct_every=corr)
    mixed = [x.clone() for x in v]
    for C in (16, 8, 1):
        for r in range(len(Ns)):
            b.set_cluster(r, C)
            v[r].copy_(v0[r])
        b.integrate(1e-3, 5, correct_every=corr)
        for x, y, z in zip(v, mixed, v0):
            assert torch.isfinite(y).all() and not torch.equal(y, z)
            assert torch.equal(x, y)
    b.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_light_blocks_do_not_crowd_the_heavy_ones(precision):
    """128 of N = 9 in clusters of one and 128 of N = 4 in clusters of two take no
    more than 1.15 times as long as the two groups one after the other."""
    steps, n = 300, 128

    def best(Ns, Cs):
        b, _ = _batch(Ns, precision)
        for r, N in enumerate(Ns):
            b.set_cluster(r, Cs[N])
        t = min(b.integrate(1e-3, steps) for _ in range(6))
        b.close()
        return t

    Cs = {4: 2, 9: 1}
    assert best([4, 9] * n, Cs) <= 1.15 * (best([4] * n, Cs) + best([9] * n, Cs))
