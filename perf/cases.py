"""The measured workloads of the library: what a user has it do, through the
public calls of paper_1912_01491_gb300, over the sizes in use.

Kinds of a case (its "kind"), all with inputs resident on the GPU:
  structure     the canonical lists of the nonzero f and d of SU(N), written
                into the caller's buffers (kernel (a))
  assemble      dense A = Q + R and K from a Kossakowski matrix and h
  rk4           classical RK4 of one dense system: FP64, FP32 storage or BF16
                storage with row scales, with the FP64 correction every
                "correct" steps
  csr_assemble  sparse assembly of the ladder and dimer models
  csr_rk4       RK4 on the sparse ladder system
  td            RK4 of the rocked dimer, Q(t) = Q0 + eps(t) Q1
  ensemble      many random Lindbladians of mixed N: assembled, then
                integrated by the batched kernels

Sizes: N = 4 .. 200 for dense systems (M = N^2 - 1), up to N = 2000 for sparse
ones.
"""
import math

import numpy as np
import torch

import paper_1912_01491_gb300 as lb

DEV = "cuda"
DT = 1e-3


def listed():
    return [
        # the structure constants of the largest dense basis: 1.7e7 triples
        {"name": "structure_n200", "kind": "structure", "N": 200},
        # one small random Lindbladian: a call of a few launches
        {"name": "assemble_n10", "kind": "assemble", "N": 10},
        # the middle size of the dense model
        {"name": "assemble_n50", "kind": "assemble", "N": 50},
        # the paper's dense size: a is 25.6 GB, A 12.8 GB
        {"name": "assemble_n200", "kind": "assemble", "N": 200},
        # a trajectory of a small system: many short steps
        {"name": "rk4_fp64_n10", "kind": "rk4", "N": 10, "precision": "fp64", "correct": 0, "steps": 1000},
        # mixed precision at the middle size: FP32 storage, FP64 correction every 50 steps
        {"name": "rk4_fp32_n50", "kind": "rk4", "N": 50, "precision": "fp32", "correct": 50, "steps": 500},
        # the same at the paper's dense size, one correction window
        {"name": "rk4_fp32_n200", "kind": "rk4", "N": 200, "precision": "fp32", "correct": 50, "steps": 50},
        # what the serving form runs for large N: BF16 storage, correction every 5 steps
        {"name": "rk4_bf16_n150", "kind": "rk4", "N": 150, "precision": "bf16", "correct": 5, "steps": 100},
        # the sparse ladder at the paper's largest N: 2.8e7 entries
        {"name": "csr_assemble_ladder_n2000", "kind": "csr_assemble", "model": "ladder", "N": 2000},
        # and its FP32 integration
        {"name": "csr_rk4_fp32_n2000", "kind": "csr_rk4", "N": 2000, "precision": "fp32", "correct": 50,
         "steps": 100},
        # the rocked dimer: a twentieth of a drive period
        {"name": "td_dimer_n400", "kind": "td", "N": 400, "steps": 1000},
        # an ensemble of random Lindbladians, N uniform in [4, 40]
        {"name": "ensemble_256", "kind": "ensemble", "count": 256, "lo": 4, "hi": 40, "precision": "fp32",
         "correct": 50, "steps": 500},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["structure", "assemble", "assemble", "rk4", "rk4", "rk4", "csr_assemble", "csr_rk4", "td",
                       "ensemble"])
    if kind == "structure":
        return {"kind": kind, "N": _log_int(rng, 4, 200)}
    if kind == "assemble":
        return {"kind": kind, "N": _log_int(rng, 4, 200)}
    if kind == "rk4":
        N = _log_int(rng, 4, 200)
        precision = rng.choice(["fp64", "fp32", "bf16"])
        correct = 0 if precision == "fp64" else rng.choice([5, 10, 50])
        # about as many steps as a tenth of a second allows at the larger sizes
        steps = max(10, min(1000, int(4.0e10 / N ** 4)))
        return {"kind": kind, "N": N, "precision": precision, "correct": correct, "steps": steps}
    if kind == "csr_assemble":
        model = rng.choice(["ladder", "dimer"])
        return {"kind": kind, "model": model, "N": _log_int(rng, 20, 2000 if model == "ladder" else 400)}
    if kind == "csr_rk4":
        precision = rng.choice(["fp64", "fp32"])
        return {"kind": kind, "N": _log_int(rng, 20, 2000), "precision": precision,
                "correct": 0 if precision == "fp64" else 50, "steps": rng.randrange(20, 101)}
    if kind == "td":
        return {"kind": kind, "N": _log_int(rng, 20, 400), "steps": rng.randrange(100, 501)}
    lo = rng.randrange(2, 21)
    return {"kind": kind, "count": rng.randrange(16, 129), "lo": lo, "hi": rng.randrange(lo, 41),
            "precision": rng.choice(["fp32", "fp32", "fp64"]), "correct": rng.choice([0, 10, 50]),
            "steps": rng.randrange(50, 201)}


# ------------------------------------------------------------------ inputs
def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * int(seed) + salt)
    return g


def _kossakowski(M, gen, chunk=4096):
    """Hermitian positive semidefinite M x M a of trace 1: the Wishart ensemble
    of up to 512 complex Gaussian jump operators."""
    r = min(M, 512)
    g = torch.randn((M, 2 * r), generator=gen, device=DEV, dtype=torch.float32)
    g /= g.double().norm().item()
    x, y = g[:, :r], g[:, r:]
    a = torch.empty((M, M), dtype=torch.complex128, device=DEV)
    v = torch.view_as_real(a)
    re_l, im_l, rhs = torch.cat([x, y], 1), torch.cat([y, -x], 1), g.T.contiguous()
    for r0 in range(0, M, chunk):
        v[r0:r0 + chunk, :, 0] = re_l[r0:r0 + chunk] @ rhs
        v[r0:r0 + chunk, :, 1] = im_l[r0:r0 + chunk] @ rhs
    for r0 in range(0, M, chunk):  # exactly Hermitian
        for c0 in range(r0, M, chunk):
            b = 0.5 * (a[r0:r0 + chunk, c0:c0 + chunk] + a[c0:c0 + chunk, r0:r0 + chunk].mH)
            a[r0:r0 + chunk, c0:c0 + chunk] = b
            a[c0:c0 + chunk, r0:r0 + chunk] = b.mH
    return a


def _level(N, k):
    """Coherence vector of |k><k| (FP64, device)."""
    v = torch.zeros(N * N - 1, dtype=torch.float64, device=DEV)
    v[N * (N - 1):] = _diagonals(N)[:, k]
    return v


def _dense_system(N, gen):
    """A and K with the make-up of a random Lindbladian's: an antisymmetric
    part of about 4N entries of order one in a row (Q of a GUE Hamiltonian)
    and a dense part of entries about M^-3/2 with -1/N on the diagonal (R of a
    Wishart Kossakowski matrix of trace 1)."""
    M = N * N - 1
    A = torch.randn((M, M), generator=gen, device=DEV, dtype=torch.float64)
    A *= 3.0 / M ** 1.5
    n = min(4 * N, M // 2)
    rows = torch.arange(M, device=DEV).repeat_interleave(n)
    cols = torch.randint(0, M, (M * n,), generator=gen, device=DEV)
    q = torch.randn(M * n, generator=gen, device=DEV, dtype=torch.float64) * math.sqrt(0.5)
    flat = A.view(-1)
    keep = rows < cols
    key = torch.unique(rows[keep] * M + cols[keep])
    q = q[:key.numel()]
    flat[key] += q
    flat[(key % M) * M + key // M] -= q
    A.diagonal().sub_(1.0 / N)
    K = torch.randn(M, generator=gen, device=DEV, dtype=torch.float64) / M
    return A, K


def _model(case, seed):
    """(H, L, rate) of the sparse models as numpy arrays; for the dimer H is
    (H0, H1)."""
    N = case["N"]
    g = np.random.default_rng(int(seed) + 17)
    if case.get("model", "ladder") == "ladder" and case["kind"] != "td":
        # real tridiagonal H, L = sum_n sqrt(n) |n-1><n|
        H = np.diag(g.uniform(-1.0, 1.0, N)) + np.diag(np.ones(N - 1), 1) + np.diag(np.ones(N - 1), -1)
        return H, np.diag(np.sqrt(np.arange(1.0, N)), 1), 0.1
    # periodically rocked Bose-Hubbard dimer of N - 1 bosons
    J, U, gamma = -1.0, float(g.uniform(1.8, 2.6)), 0.1
    n = np.arange(N, dtype=np.float64)
    hop = np.diag(np.sqrt((n[:-1] + 1.0) * (N - 1.0 - n[:-1])), -1)
    n1, n2 = n, N - 1.0 - n
    H0 = -J * (hop + hop.T) + np.diag(2.0 * U / (N - 1.0) * (n1 * (n1 - 1.0) + n2 * (n2 - 1.0)))
    return (H0, np.diag(n2 - n1)), np.diag(n1 - n2) - hop + hop.T, gamma / (N - 1.0)


EPS = (-2.5, 0.5)          # the dimer's drive on the two halves of its period
PERIOD = 2.0 * math.pi
TD_STEPS = 20000           # steps of one period


def _dev(x):
    return torch.tensor(np.ascontiguousarray(x), dtype=torch.complex128, device=DEV)


def _sparse_inputs(B, H, L, rate):
    l = B.expand(_dev(L))
    nz = torch.nonzero(l.abs() > 0).flatten()
    return B.expand(_dev(H)).real.contiguous(), [(rate, nz, l[nz].contiguous())]


def _state0(case, seed):
    """Coherence vector the sparse models start from."""
    N = case["N"]
    return _level(N, N - 1 - int(seed) % 2)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "structure":
        # the caller's buffers, a little larger than the lists and full of other work's
        # values, which stay past the lists' ends
        s["B"] = lb.Basis(case["N"])
        s["f"], s["d"] = _buffers(case["N"], seed)
    elif kind == "assemble":
        B = s["B"] = lb.Basis(case["N"])
        g = _gen(seed, 2)
        s["a"] = _kossakowski(B.M, g)
        s["h"] = torch.randn(B.M, generator=g, device=DEV, dtype=torch.float64)  # GUE Hamiltonian
        s["A"] = torch.empty((B.M, B.M), dtype=torch.float64, device=DEV)
        s["K"] = torch.empty(B.M, dtype=torch.float64, device=DEV)
    elif kind == "rk4":
        N = case["N"]
        A, K = _dense_system(N, _gen(seed, 3))
        s["K"], s["v0"], s["A64"], s["scale"] = K, _level(N, int(seed) % N), None, None
        if case["precision"] == "fp64":
            s["Ap"] = A
        else:
            s["A64"] = A
            if case["precision"] == "fp32":
                s["Ap"] = lb.pack_fp32(A)
            else:
                s["Ap"], s["scale"] = lb.pack_bf16(A)
        s["work"] = lb.rk4_workspace(N * N - 1, DEV)
    elif kind == "csr_assemble":
        H, L, rate = _model(case, seed)
        B = s["B"] = lb.Basis(case["N"])
        s["h"], s["channels"] = _sparse_inputs(B, H if case["model"] == "ladder" else H[0], L, rate)
    elif kind == "csr_rk4":
        H, L, rate = _model(case, seed)
        B = lb.Basis(case["N"])
        h, ch = _sparse_inputs(B, H, L, rate)
        s["csr"], s["v0"] = lb.Csr(B, h=h, channels=ch), _state0(case, seed)
        s["work"] = lb.rk4_workspace(B.M, DEV)
    elif kind == "td":
        (H0, H1), L, rate = _model(case, seed)
        B = lb.Basis(case["N"])
        h, ch = _sparse_inputs(B, H0, L, rate)
        s["A0"] = lb.Csr(B, h=h, channels=ch)
        s["Q1"] = lb.Csr(B, h=B.expand(_dev(H1)).real.contiguous(), channels=())
        s["v0"] = _state0(case, seed)
        s["work"] = lb.rk4_workspace(B.M, DEV)
    else:
        Ns = _sizes(case)
        g = _gen(seed, 4)
        b = s["batch"] = lb.Batch(Ns)
        M = [n * n - 1 for n in Ns]
        s["v0"] = torch.cat([_level(n, r % n) for r, n in enumerate(Ns)])
        s["v"] = s["v0"].clone()
        for r, v in enumerate(s["v"].split(M)):
            b.set(r, _kossakowski(M[r], g), torch.randn(M[r], generator=g, device=DEV, dtype=torch.float64), v)
        b.set_precision(case["precision"])
        b.assemble("closed")
        b.tune(width=6, probe_steps=20, dt=DT)  # cluster sizes, once for the ensemble's sizes
        s["v"].copy_(s["v0"])
    return s


def _buffers(N, seed):
    """(indices, values) for the lists of f and of d."""
    g = _gen(seed, 1)
    return [(torch.randint(-9, 0, (n + 16, 3), generator=g, device=DEV, dtype=torch.int32),
             torch.randn(n + 16, generator=g, device=DEV, dtype=torch.float64)) for n in _structure_counts(N)]


def _sizes(case):
    """N of every realization; the same for every seed of a case."""
    return [int(n) for n in np.random.default_rng(7).integers(case["lo"], case["hi"] + 1, case["count"])]


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "structure":
        out = []
        for w in "fd":
            idx, val = s[w]
            out += [idx, val, s["B"].structure_into(w, idx, val)]
        return out
    if kind == "assemble":
        out = s["B"].assemble_dense(s["a"], h=s["h"], A=s["A"], K=s["K"])
        return [out["A"], out["K"]]
    if kind == "rk4":
        v = s["v0"].clone()
        lb.rk4_dense(s["Ap"], s["K"], v, DT, case["steps"], precision=case["precision"], scale=s["scale"],
                     A64=s["A64"], correct_every=case["correct"], work=s["work"])
        return v
    if kind == "csr_assemble":
        c = lb.Csr(s["B"], h=s["h"], channels=s["channels"])
        return list(_csr_tensors(c)) + [c.nnz]
    if kind == "csr_rk4":
        v = s["v0"].clone()
        s["csr"].rk4(v, _csr_dt(case), case["steps"], precision=case["precision"], correct_every=case["correct"],
                     work=s["work"])
        return v
    if kind == "td":
        v = s["v0"].clone()
        s["A0"].rk4_td(s["Q1"], v, PERIOD / TD_STEPS, case["steps"], [0.0, PERIOD / 2], list(EPS), PERIOD,
                       t0=_td_start(case), work=s["work"])
        return v
    s["v"].copy_(s["v0"])
    s["batch"].assemble("closed")
    s["batch"].integrate(DT, case["steps"], correct_every=case["correct"])
    return s["v"]


def _csr_dt(case):
    # the damping of the ladder's levels grows as N
    return DT * min(1.0, 500.0 / case["N"])


def _td_start(case):
    # the drive switches within the run
    return PERIOD / 2 - PERIOD / TD_STEPS * (case["steps"] // 2)


class _Array:
    """A device array of a sparse system, as torch sees it."""

    def __init__(self, owner, ptr, n, kind):
        self.owner = owner  # the arrays belong to the system
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": kind, "data": (ptr, False), "version": 3}


def _csr_tensors(c):
    """(row pointers, columns, values, K) of a sparse system, in place on the device."""
    import ctypes
    p = [ctypes.c_void_p() for _ in range(4)]
    if lb.native.load().lb_csr_arrays(c._h, *[ctypes.byref(x) for x in p]) != 0:
        raise RuntimeError("lb_csr_arrays")
    kinds = ((c.M + 1, "<i8"), (c.nnz, "<i4"), (c.nnz, "<f8"), (c.M, "<f8"))
    return [torch.as_tensor(_Array(c, x.value, n, k), device=DEV) for x, (n, k) in zip(p, kinds)]


# ------------------------------------------------------------------ work
def _structure_counts(N):
    """Canonical nonzeros of f and d."""
    tri = N * (N - 1) * (N - 2) // 6
    f = 4 * tri + sum((b - max(a, 1) + 1) for a in range(N) for b in range(a + 1, N))
    d = 4 * tri + 2 * (sum(N - max(a, 1) for a in range(N) for _ in range(a + 1, N)) - 1) + N * (N - 1) // 2 - 1
    return f, d


def _csr_entries(case):
    N = case["N"]
    if case["kind"] == "csr_rk4" or case.get("model") == "ladder":
        return 7 * N * N - 11 * N + 1
    return 18 * N * N  # the dimer's A0, about


def work(case):
    kind = case["kind"]
    if kind == "structure":
        n = sum(_structure_counts(case["N"]))
        return {"bytes": 20 * n, "flops": 0}
    if kind == "assemble":
        M = case["N"] ** 2 - 1
        # one triangle of the Hermitian a, A, h, K; the eight terms of a pair x pair entry
        return {"bytes": 8 * M * M + 8 * M * M + 16 * M, "flops": 8 * M * M}
    if kind == "rk4":
        M = case["N"] ** 2 - 1
        esz = {"fp64": 8, "fp32": 4, "bf16": 2}[case["precision"]]
        n, c = case["steps"], case["correct"]
        corr = -(-n // c) if c else 0
        return {"bytes": _streamed(esz * M * M, 4 * n) + _streamed((8 + esz) * M * M, corr) + 4 * n * 40 * M,
                "flops": 8 * M * M * n + corr * 3 * M * M}
    if kind == "csr_assemble":
        M, nnz = case["N"] ** 2 - 1, _csr_entries(case)
        return {"bytes": 12 * nnz + 24 * M, "flops": 2 * nnz}
    if kind == "csr_rk4":
        M, nnz = case["N"] ** 2 - 1, _csr_entries(case)
        esz = 8 if case["precision"] == "fp64" else 4
        n = case["steps"]
        return {"bytes": _streamed((esz + 4) * nnz + 8 * M, 4 * n) + 4 * n * 36 * M, "flops": 8 * nnz * n}
    if kind == "td":
        M, nnz = case["N"] ** 2 - 1, _csr_entries(case) + 2 * case["N"] ** 2
        n = case["steps"]
        return {"bytes": _streamed(12 * nnz + 16 * M, 4 * n) + 4 * n * 40 * M, "flops": 8 * nnz * n}
    esz = 8 if case["precision"] == "fp64" else 4
    m2 = sum((n * n - 1) ** 2 for n in _sizes(case))
    return {"bytes": 16 * m2 + esz * m2, "flops": 8 * m2 * (1 + case["steps"])}


def _streamed(size, times):
    """Bytes a matrix of `size` costs when it is read `times` times: once, if
    it stays on the chip (126 MB of L2)."""
    return size * times if size > 126e6 else size


# ------------------------------------------------------------------ values in 64 bits, without the library
def _diagonals(N):
    """(N - 1) x N: the diagonals of D_1 .. D_{N-1}."""
    l = torch.arange(1, N, dtype=torch.float64, device=DEV)[:, None]
    k = torch.arange(N, dtype=torch.float64, device=DEV)[None, :]
    return torch.where(k < l, torch.ones_like(k), torch.where(k == l, -l, torch.zeros_like(k))) / torch.sqrt(
        l * (l + 1.0))


def _pairs(N):
    return torch.triu_indices(N, N, 1, device=DEV)


def _to_units(X, N):
    """sum_j X[j] (F_j)_pq along the first axis: M rows to N^2 rows (p, q)."""
    P = N * (N - 1) // 2
    a, b = _pairs(N)
    Y = torch.empty((N * N,) + X.shape[1:], dtype=torch.complex128, device=DEV)
    r = math.sqrt(0.5)
    Y[a * N + b] = r * (X[:P] - 1j * X[P:2 * P])
    Y[b * N + a] = r * (X[:P] + 1j * X[P:2 * P])
    Y[torch.arange(N, device=DEV) * (N + 1)] = _diagonals(N).T.to(torch.complex128) @ X[2 * P:].to(torch.complex128)
    return Y


def _traces(Y, N):
    """Tr(F_s Y) along the first axis: N^2 rows (p, q) to M rows."""
    P = N * (N - 1) // 2
    a, b = _pairs(N)
    X = torch.empty((N * N - 1,) + Y.shape[1:], dtype=torch.complex128, device=DEV)
    r = math.sqrt(0.5)
    ab, ba = Y[a * N + b], Y[b * N + a]
    X[:P] = r * (ab + ba)
    X[P:2 * P] = 1j * r * (ab - ba)
    X[2 * P:] = _diagonals(N).to(torch.complex128) @ Y[torch.arange(N, device=DEV) * (N + 1)]
    return X


def _generator(N, a, h):
    """(A, K): the generator applied to the matrix units, back in the basis."""
    X = _to_units(a, N)
    X = _to_units(X.T.contiguous(), N).T.contiguous()  # [(p, q), (p', q')], sum of a_jk (F_j)_pq (F_k)_p'q'
    X = X.view(N, N, N, N)
    G = torch.einsum("pqrp->rq", X)                    # sum a_jk F_k F_j
    S = X.permute(0, 3, 1, 2).contiguous()             # out (p, q'), in (q, p')
    del X
    H = _to_units(h.to(torch.complex128), N).view(N, N)
    left, right = -0.5 * G - 1j * H, -0.5 * G + 1j * H  # left rho + rho right
    i = torch.arange(N, device=DEV)
    S[:, i, :, i] += left
    S[i, :, i, :] += right.T
    S = S.view(N * N, N * N)
    K = _traces(S @ torch.eye(N, dtype=torch.complex128, device=DEV).view(-1) / N, N).real
    S = _traces(S, N)
    # columns: A_sn = sum over the units of S[s, (q, p')] (F_n)_(q, p')
    P = N * (N - 1) // 2
    pa, pb = _pairs(N)
    A = torch.empty((N * N - 1, N * N - 1), dtype=torch.float64, device=DEV)
    r = math.sqrt(0.5)
    ab, ba = S[:, pa * N + pb], S[:, pb * N + pa]
    A[:, :P] = r * (ab + ba).real
    A[:, P:2 * P] = r * (ab - ba).imag
    A[:, 2 * P:] = S[:, i * (N + 1)].real @ _diagonals(N).T
    return A, K


def _rk4(f, v, dt, steps, t0=0.0):
    for n in range(steps):
        t = t0 + n * dt
        k1 = f(v, t + 1e-6 * dt)
        k2 = f(v + 0.5 * dt * k1, t + 0.5 * dt)
        k3 = f(v + 0.5 * dt * k2, t + 0.5 * dt)
        k4 = f(v + dt * k3, t + dt - 1e-6 * dt)
        v = v + dt / 6.0 * (k1 + 2.0 * (k2 + k3) + k4)
    return v


def _structure_exact(N):
    """(f values, d values) in the order of the lists: triples m <= n <= s."""
    P = N * (N - 1) // 2
    out = []
    c = [0.0] + [1.0 / math.sqrt(l * (l + 1.0)) for l in range(1, N)]
    c = torch.tensor(c, dtype=torch.float64, device=DEV)
    pidx = torch.zeros((N, N), dtype=torch.int64, device=DEV)
    pa, pb = _pairs(N)
    pidx[pa, pb] = torch.arange(P, device=DEV)
    tri = torch.combinations(torch.arange(N, device=DEV), 3)
    x, y, z = tri[:, 0], tri[:, 1], tri[:, 2]
    e = [pidx[x, y], pidx[y, z], pidx[x, z]]  # T = c(x->y) c(y->z) c(z->x)
    D = _diagonals(N)
    for w in "fd":
        keys, vals = [], []

        def add(i, j, k, v):
            t = torch.sort(torch.stack([i, j, k]), 0).values
            keys.append((t[0] * N * N + t[1]) * N * N + t[2])
            vals.append(v.expand(t.shape[1]) if v.dim() == 0 else v)

        for kinds in range(8):
            t = [(kinds >> q) & 1 for q in range(3)]
            if sum(t) % 2 != (1 if w == "f" else 0) or tri.shape[0] == 0:
                continue
            # J carries -i along the rising direction, +i along z -> x
            T = (1j if t[2] else 1.0) * (-1j if t[0] else 1.0) * (-1j if t[1] else 1.0) * 0.5 * math.sqrt(0.5)
            T = complex(T)
            # f of the sorted triple: 2 Im Tr(F_s F_m F_n), the sign of the order of the three
            idx = torch.stack([e[q] + t[q] * P for q in range(3)])
            order = torch.argsort(idx, 0)
            even = (order[1] - order[0]) % 3 == 1
            v = torch.where(even, 1.0, -1.0).double() * (2.0 * T.imag) if w == "f" else torch.tensor(
                2.0 * T.real, dtype=torch.float64, device=DEV)
            add(idx[0], idx[1], idx[2], v)
        e2 = torch.arange(P, device=DEV)
        for l in range(1, N):
            da, db = D[l - 1][pa], D[l - 1][pb]
            dl = torch.full_like(e2, 2 * P + l - 1)
            if w == "f":
                v = da - db  # f(S_ab, J_ab, D_l)
                k = (pa <= l) & (l <= pb) & (l >= 1)
                add(e2[k], e2[k] + P, dl[k], v[k])
            else:
                v = da + db
                k = (pa <= l) & ~((pa == 0) & (pb == 1) & (l == 1))
                add(e2[k], e2[k], dl[k], v[k])
                add(e2[k] + P, e2[k] + P, dl[k], v[k])
        if w == "d":
            l, r = torch.triu_indices(N - 1, N - 1, device=DEV) + 1
            k = ~((l == 1) & (r == 1))
            l, r = l[k], r[k]
            v = torch.where(l == r, 2.0 * (1.0 - l.double()) * c[l], 2.0 * c[r])
            add(2 * P + l - 1, 2 * P + l - 1, 2 * P + r - 1, v)
        key, val = torch.cat(keys), torch.cat(vals)
        out.append(val[torch.argsort(key)])
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "structure":
        out = []
        for v, (_, rest) in zip(_structure_exact(case["N"]), _buffers(case["N"], seed)):
            out += [None, torch.cat([v, rest[v.numel():]]), None]
        return out
    if kind == "assemble":
        g = _gen(seed, 2)
        M = case["N"] ** 2 - 1
        a = _kossakowski(M, g)
        h = torch.randn(M, generator=g, device=DEV, dtype=torch.float64)
        return list(_generator(case["N"], a, h))
    if kind == "rk4":
        N = case["N"]
        A, K = _dense_system(N, _gen(seed, 3))
        return _rk4(lambda v, t: A @ v + K, _level(N, int(seed) % N), DT, case["steps"])
    if kind == "csr_assemble":
        N = case["N"]
        if N > 64:
            return None
        H, L, rate = _model(case, seed)
        H = H if case["model"] == "ladder" else H[0]
        l = _traces(_dev(L).view(-1), N)
        h = _traces(_dev(H).view(-1), N).real
        A, K = _generator(N, rate * torch.outer(l, l.conj()), h)
        return [None, None, A[A.abs() > 1e-11 * A.abs().max()], K, None]
    if kind in ("csr_rk4", "td"):
        N = case["N"]
        H, L, rate = _model(case, seed)
        H0, H1 = (_dev(H), None) if kind == "csr_rk4" else (_dev(H[0]), _dev(H[1]))
        if N > 500:
            return _ladder_exact(case, seed, H, L, rate)
        L = _dev(L)
        LL = 0.5 * L.mH @ L

        def f(rho, t):
            h = H0 if H1 is None else H0 + (EPS[0] if t % PERIOD < PERIOD / 2 else EPS[1]) * H1
            x = (-1j * h - rate * LL) @ rho
            return x + x.mH + rate * (L @ rho @ L.mH)

        rho = torch.zeros((N, N), dtype=torch.complex128, device=DEV)
        k = N - 1 - int(seed) % 2
        rho[k, k] = 1.0
        dt, t0 = (_csr_dt(case), 0.0) if kind == "csr_rk4" else (PERIOD / TD_STEPS, _td_start(case))
        return _traces(_rk4(f, rho, dt, case["steps"], t0).reshape(-1), N).real
    Ns = _sizes(case)
    g = _gen(seed, 4)
    out = []
    for r, n in enumerate(Ns):
        a = _kossakowski(n * n - 1, g)
        h = torch.randn(n * n - 1, generator=g, device=DEV, dtype=torch.float64)
        A, K = _generator(n, a, h)
        # one step is v + dt (D v + c): the four stages of a linear system with constant A and K
        D, k, one = A, K, DT
        for q in (4.0, 3.0, 2.0):
            D, k = A + (one / q) * (A @ D), K + (one / q) * (A @ k)
        v = _level(n, r % n)
        for _ in range(case["steps"]):
            v = v + one * (D @ v + k)
        out.append(v)
    return torch.cat(out)


def _ladder_exact(case, seed, H, L, rate):
    """The ladder on rho itself, its two bands applied element by element."""
    N = case["N"]
    d = torch.tensor(np.diag(H), device=DEV)
    w = torch.tensor(np.diag(L, 1), device=DEV)  # sqrt(n), n = 1 .. N - 1
    n = torch.arange(N, dtype=torch.float64, device=DEV)

    def f(rho, t):
        x = (d[:, None] - d[None, :]) * rho
        x[1:] += rho[:-1]
        x[:-1] += rho[1:]
        x[:, 1:] -= rho[:, :-1]
        x[:, :-1] -= rho[:, 1:]
        y = -1j * x - (0.5 * rate) * (n[:, None] + n[None, :]) * rho
        y[:-1, :-1] += rate * (w[:, None] * w[None, :]) * rho[1:, 1:]
        return y

    rho = torch.zeros((N, N), dtype=torch.complex128, device=DEV)
    k = N - 1 - int(seed) % 2
    rho[k, k] = 1.0
    return _traces(_rk4(f, rho, _csr_dt(case), case["steps"]).reshape(-1), N).real
