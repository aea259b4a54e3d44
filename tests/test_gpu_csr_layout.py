"""The layout of sparse systems by groups of 32 rows (lb_csr_reg.cu; needs an
sm_103a GPU) against the plain FP64 product of the CSR arrays on the host."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_01491_gb300 import build
    build.build()


def _system(B, model, seed):
    import paper_1912_01491_gb300 as lb
    N = B.N
    Q1 = None
    if model == "ladder":
        H, L, g = wl.ladder_model(N, seed)
    elif model == "dimer":
        H, H1, L, g, _ = wl.dimer_model(N)
        Q1 = lb.Csr(B, h=B.expand(torch.tensor(H1, device="cuda")).real.contiguous(), channels=())
    else:  # a few random matrix elements: no two rows alike, some of them long
        r = np.random.default_rng(seed)
        H, L, g = np.zeros((N, N), complex), np.zeros((N, N), complex), 0.7
        for m in (H, L):
            m[r.integers(0, N, N), r.integers(0, N, N)] = r.standard_normal(N) + 1j * r.standard_normal(N)
        H = H + H.conj().T
    l = B.expand(torch.tensor(L, device="cuda"))
    nz = torch.nonzero(l.abs() > 0).flatten()
    h = B.expand(torch.tensor(H, device="cuda")).real.contiguous()
    return lb.Csr(B, h=h, channels=[(g, nz, l[nz].contiguous())]), Q1


def _dense(c):
    rp, col, val, K = c.to_host()
    A = np.zeros((c.M, c.M))
    for s in range(c.M):
        A[s, col[rp[s]:rp[s + 1]]] = val[rp[s]:rp[s + 1]]
    return A, K


def _rk4(f, v, dt, steps):
    for _ in range(steps):
        k1 = f(v)
        k2 = f(v + 0.5 * dt * k1)
        k3 = f(v + 0.5 * dt * k2)
        k4 = f(v + dt * k3)
        v = v + dt / 6.0 * (k1 + 2 * k2 + 2 * k3 + k4)
    return v


# systems of one group, of a last group that is not whole, of only explicit groups (small N) and of mostly regular
# ones; the random model has rows of any length
@pytest.mark.parametrize("model,N", [("ladder", 2), ("ladder", 5), ("ladder", 6), ("ladder", 24), ("ladder", 71),
                                     ("dimer", 4), ("dimer", 17), ("dimer", 50), ("random", 9), ("random", 30)])
def test_stages_against_the_csr_product(model, N):
    """FP64 within 1e-13 of the host's (7 steps of sums of at most M terms),
    FP32 storage with the correction within 1e-6, and the driven form with a
    constant drive equal to its matrix A0 + eps Q1."""
    import paper_1912_01491_gb300 as lb
    with lb.Basis(N) as B:
        c, Q1 = _system(B, model, 3 * N)
        A, K = _dense(c)
        v0 = np.random.default_rng(N).standard_normal(c.M)
        dt, steps = 0.2 / max(1.0, np.abs(A).sum(1).max()), 7
        ref = _rk4(lambda v: A @ v + K, v0, dt, steps)
        raw = torch.zeros(c.M + 1, dtype=torch.float64, device="cuda")
        for off in (0, 1):  # the state 8 bytes off 16-byte alignment
            v = raw[off:off + c.M]
            v.copy_(torch.tensor(v0))
            c.rk4(v, dt, steps)
            assert np.linalg.norm(v.cpu().numpy() - ref) <= 1e-13 * np.linalg.norm(ref)
        v = torch.tensor(v0, device="cuda")
        c.rk4(v, dt, steps, precision="fp32", correct_every=3)
        assert np.linalg.norm(v.cpu().numpy() - ref) <= 1e-6 * np.linalg.norm(ref)
        if Q1 is not None:
            A1, _ = _dense(Q1)
            eps = -0.8
            ref = _rk4(lambda v: (A + eps * A1) @ v + K, v0, dt, steps)
            v = torch.tensor(v0, device="cuda")
            c.rk4_td(Q1, v, dt, steps, [0.0], [eps], 1.0)
            assert np.linalg.norm(v.cpu().numpy() - ref) <= 1e-13 * np.linalg.norm(ref)
            Q1.close()
        c.close()


def test_two_streams_share_one_system():
    """The layout is made once; integrations of one system on two streams give
    the same bits."""
    import paper_1912_01491_gb300 as lb
    with lb.Basis(60) as B:
        c, _ = _system(B, "ladder", 1)
        v0 = torch.tensor(np.random.default_rng(0).standard_normal(c.M), device="cuda")
        torch.cuda.synchronize()
        out = []
        for _ in range(2):
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                v = v0.clone()
                c.rk4(v, 1e-3, 20, work=lb.rk4_workspace(c.M), stream=s)
            out.append(v)
        torch.cuda.synchronize()
        assert torch.equal(out[0], out[1]) and not torch.equal(out[0], v0)
        c.close()
