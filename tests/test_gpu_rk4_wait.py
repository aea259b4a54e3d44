"""A wait between the blocks of the one-launch RK4 (lb_rk4_persist.cu; needs an
sm_103a GPU) that runs out: with a limit below zero a block gives up where a
word has not come yet.  The launch ends, lb_integrate returns LB_ETIMEOUT and
writes nothing, the asynchronous form leaves NaN, and the next call is right."""
import ctypes

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


class _Limit:
    def __init__(self, cycles):
        from paper_1912_01491_gb300 import native
        self.f = native.load().lbi_poll_cycles
        self.f.restype, self.f.argtypes = ctypes.c_longlong, [ctypes.c_longlong]
        self.cycles = cycles

    def __enter__(self):
        self.before = self.f(self.cycles)

    def __exit__(self, *exc):
        self.f(self.before)


def _system(M):
    g = torch.Generator(device="cuda")
    g.manual_seed(M)
    A = torch.randn((M, M), generator=g, device="cuda", dtype=torch.float64) / M ** 0.5
    return A, torch.randn(M, generator=g, device="cuda", dtype=torch.float64) / M


@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("M", [99, 1680, 3400])
def test_every_element_is_right_or_nan(M, precision):
    import paper_1912_01491_gb300 as lb
    A, K = _system(M)
    Ap, scale = (A, None) if precision == "fp64" else (lb.pack_fp32(A), None) if precision == "fp32" else lb.pack_bf16(A)
    v0 = torch.linspace(-1, 1, M, dtype=torch.float64, device="cuda")
    kw = dict(precision=precision, scale=scale, A64=None if precision == "fp64" else A,
              correct_every=0 if precision == "fp64" else 3, snap_every=4)
    steps = 40
    right, v = v0.clone(), v0.clone()
    s_right = lb.rk4_dense(Ap, K, right, 1e-2, steps, **kw)
    with _Limit(-1):
        s = lb.rk4_dense(Ap, K, v, 1e-2, steps, **kw)
    torch.cuda.synchronize()
    assert torch.isfinite(s_right).all() and torch.isnan(v).all()
    assert (torch.isnan(s) | (s == s_right)).all() and torch.isnan(s[-1]).all()
    v = v0.clone()
    lb.rk4_dense(Ap, K, v, 1e-2, steps, **kw)
    assert torch.equal(v, right)


@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("M", [1, 33, 257, 2499])
def test_a_nan_reaches_every_row_in_one_step(M, precision):
    """What one block sends instead of a value it could not form: also through
    the padding of the rows and past the products with zero elements."""
    import paper_1912_01491_gb300 as lb
    A, K = _system(M)
    A[:, M // 2] = 0.0
    Ap, scale = (A, None) if precision == "fp64" else (lb.pack_fp32(A), None) if precision == "fp32" else lb.pack_bf16(A)
    v = torch.ones(M, dtype=torch.float64, device="cuda")
    v[M // 2] = float("nan")
    lb.rk4_dense(Ap, K, v, 1e-2, 1, precision=precision, scale=scale)
    assert torch.isnan(v).all()


@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16"])
def test_host_calls_return_the_timeout(precision):
    import paper_1912_01491_gb300 as lb
    from paper_1912_01491_gb300 import native
    N = 12
    M = N * N - 1
    r = np.random.default_rng(2)
    G = r.standard_normal((M, M)) + 1j * r.standard_normal((M, M))
    with lb.Basis(N) as B:
        s = lb.System(B, a=G @ G.conj().T / M ** 2)
        v0 = r.standard_normal(M) * 0.1
        kw = dict(precision=precision, correct_every=0 if precision == "fp64" else 4)
        right = s.integrate(v0, 0.02, 1e-3, **kw)
        for snap in (0, 5):
            out = np.full((4, M) if snap else (M,), 7.0)
            with _Limit(-1), pytest.raises(lb.LBError) as ei:
                s.integrate(v0, 0.02, 1e-3, snap_every=snap, out=out, **kw)
            assert ei.value.code == native.LB_ETIMEOUT and (out == 7.0).all()
        v = v0.copy()
        with _Limit(-1), pytest.raises(lb.LBError) as ei:
            s.integrate_resume(v, 1e-3, 20, **kw)
        assert ei.value.code == native.LB_ETIMEOUT and np.array_equal(v, v0)
        assert np.array_equal(s.integrate(v0, 0.02, 1e-3, **kw), right)
        s.close()
