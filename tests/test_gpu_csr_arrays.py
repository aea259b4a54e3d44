"""RK4 on the CSR arrays of sparse systems whose rows do not suit the layout by
groups of 32 (needs an sm_103a GPU): the pipelined and the block-staged stage for
short rows, the stages with several lanes a row, and the driven ones, against
FP64 products on the host.  The numbers of launches show which kernels ran."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
sp = pytest.importorskip("scipy.sparse")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_01491_gb300 import build
    build.build()


def _system(B, k, spread, ladder):
    """H full on k levels, diagonal elsewhere: spread over all levels, one or two
    rows of a group of 32 are much longer than the rest (padding); on the first
    k of few levels, more than an eighth of the rows is long."""
    import paper_1912_01491_gb300 as lb
    N = B.N
    r = np.random.default_rng(N + k)
    H = np.diag(r.standard_normal(N)).astype(complex)
    X = r.standard_normal((k, k))
    lev = np.arange(k) * (N // k) if spread else np.arange(k)
    H[np.ix_(lev, lev)] += X + X.T
    L = np.diag(np.where(np.arange(N) < N // 2, 1.0, 0.3)).astype(complex)
    if ladder:
        L = np.diag(np.sqrt(np.arange(1.0, N)), 1).astype(complex)
    l = B.expand(torch.tensor(L, device="cuda"))
    nz = torch.nonzero(l.abs() > 1e-14).flatten()
    h = B.expand(torch.tensor(H, device="cuda")).real.contiguous()
    return lb.Csr(B, h=h, channels=[(0.1, nz, l[nz].contiguous())])


def _matrix(c):
    rp, col, val, K = c.to_host()
    return sp.csr_matrix((val, col, rp), shape=(c.M, c.M)), K


def _rk4(f, v, dt, steps):
    for _ in range(steps):
        k1 = f(v)
        k2 = f(v + 0.5 * dt * k1)
        k3 = f(v + 0.5 * dt * k2)
        k4 = f(v + dt * k3)
        v = v + dt / 6.0 * (k1 + 2 * k2 + 2 * k3 + k4)
    return v


def _launches(f):
    import paper_1912_01491_gb300 as lb
    n = lb.native.launch_count()
    f()
    return lb.native.launch_count() - n


def _width(c):
    w = 1
    while w < 32 and 4 * 2 * w <= c.nnz / c.M:
        w *= 2
    return w


# one lane a row, one chunk of 256 rows a block and several (N = 800: the buffers of the pipelined stage are reused and
# the parity flips); 4 and 8 lanes a row
CASES = [(60, 6, True, False, 1), (80, 8, True, True, 1), (800, 8, True, False, 1), (40, 20, False, False, 4),
         (40, 24, False, True, 8)]


@pytest.mark.parametrize("N,k,spread,ladder,width", CASES)
def test_stages_on_the_csr_arrays(N, k, spread, ladder, width):
    """FP64 within 1e-13 of the host's (7 steps), FP32 storage with the correction
    within 1e-6; the same bits whatever the alignment of v."""
    import paper_1912_01491_gb300 as lb
    with lb.Basis(N) as B:
        c, c32 = _system(B, k, spread, ladder), _system(B, k, spread, ladder)
        assert _width(c) == width
        A, K = _matrix(c)
        v0 = np.random.default_rng(N).standard_normal(c.M)
        dt, steps = 0.2 / max(1.0, abs(A).sum(1).max()), 7
        ref = _rk4(lambda v: A @ v + K, v0, dt, steps)
        raw = torch.zeros(c.M + 1, dtype=torch.float64, device="cuda")
        work = lb.rk4_workspace(c.M)
        for m, prec, ce, bar in ((c, "fp64", 0, 1e-13), (c32, "fp32", 3, 1e-6)):
            got, n = [], []
            for off in (0, 0, 1):  # the first call of a handle, a later one, the state 8 bytes off 16-byte alignment
                v = raw[off:off + c.M]
                v.copy_(torch.tensor(v0))
                n.append(_launches(lambda: m.rk4(v, dt, steps, precision=prec, correct_every=ce, work=work)))
                got.append(v.cpu().numpy())
            assert np.linalg.norm(got[0] - ref) <= bar * np.linalg.norm(ref)
            assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2])
            # the layout looked at and refused: one launch (three make it); wide FP32 rows have none; FP32: the values packed
            assert n[0] - n[1] == (1 if prec == "fp64" else 2 if width == 1 else 1)
            # the pipelined stage looks for the largest chunk first, the block-staged one does not
            assert n[1] - n[2] == (1 if width == 1 else 0)
        c.close()
        c32.close()


@pytest.mark.parametrize("N,k,spread,ladder,width", [x for x in CASES if x[0] < 800])
def test_driven_stages_on_the_csr_arrays(N, k, spread, ladder, width):
    """A drive that changes at every second step, within 1e-13 of the host's."""
    import paper_1912_01491_gb300 as lb
    with lb.Basis(N) as B:
        c = _system(B, k, spread, ladder)
        H1 = np.diag(np.sin(1.0 + np.arange(N))).astype(complex)
        q = lb.Csr(B, h=B.expand(torch.tensor(H1, device="cuda")).real.contiguous(), channels=())
        (A, K), (A1, _) = _matrix(c), _matrix(q)
        v0 = np.random.default_rng(N).standard_normal(c.M)
        steps, eps = 8, (0.7, -0.4)
        dt = 0.2 / max(1.0, (abs(A) + abs(A1)).sum(1).max())
        ref = v0
        for s in range(0, steps, 2):
            m = A + eps[(s // 2) % 2] * A1
            ref = _rk4(lambda v: m @ v + K, ref, dt, 2)
        n = []
        for _ in range(2):
            v = torch.tensor(v0, device="cuda")
            n.append(_launches(lambda: c.rk4_td(q, v, dt, steps, [0.0, 2 * dt], list(eps), 4 * dt)))
            assert np.linalg.norm(v.cpu().numpy() - ref) <= 1e-13 * np.linalg.norm(ref)
        assert n[0] - n[1] == 1 and n[1] == 4 * steps
        c.close()
        q.close()
