"""The work that a user of this framework has it do, as cases that can be timed and compared.

Every case is one evaluation (total cost and its exact gradient with respect to every control) of a
control problem, or one launch of a batch of them, through the package's public entry points.  The
systems are those of the repository's own workloads and benchmark: coupled qubits and transmons, a
transmon and a cavity, qubits with a random drift, and the lab-frame cat-state system.

The FP64 form is called as the optimiser loop calls it, from host memory.  The FP32 and BF16_SPLIT
forms are called as a PyTorch program calls them, whose controls are float32 parameters on the GPU:
the controls are widened into the double buffer that the entry points take, and the gradient goes
back to the parameters' type, which holds all the digits that those forms compute.
"""
import math

import numpy as np
import torch

import paper_1612_04929_gb300 as qoc

TWO_PI = 2.0 * math.pi


# ------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------
def _case(system, dims, N, precision, entry, *, dt, M=2, E=1, graph=False, propagation="unitary",
          exponential="taylor", count=1):
    return {"system": system, "dims": dims, "N": N, "M": M, "E": E, "dt": dt, "precision": precision,
            "entry": entry, "graph": graph, "propagation": propagation, "exponential": exponential,
            "count": count}


def listed():
    named = [
        # the smallest call: a two-qubit CNOT pulse of 200 slices inside a host optimiser (latency)
        ("cnot_d4_fp64", _case("zz", "2x2", 200, "fp64", "host", dt=0.5, M=4)),
        # the optimiser loop's own workload: the CNOT of two five-level transmons, four columns
        ("transmon_cnot_d25_fp64", _case("coupled", "5x5", 250, "fp64", "host", dt=0.04, M=5)),
        # a small gate trained by torch: forward and backward through autograd, four qubits
        ("qubits_d16_fp32_autograd", _case("qubits", "2x2x2x2", 2000, "fp32", "autograd", dt=0.5, M=4)),
        # the benchmark's headline: state transfer of a transmon and a cavity, replayed from its graph
        ("cavity_d40_fp32", _case("cavity", "4x10", 2000, "fp32", "device", dt=1.0, graph=True)),
        # an odd size with a detuning ensemble: three three-level transmons, the qubit subspace's columns
        ("transmons_d27_E5_fp32", _case("transmons", "3x3x3", 777, "fp32", "device", dt=0.5, M=6, E=5)),
        # a six-qubit gate, all columns
        ("qubits_d64_fp32", _case("qubits", "2x2x2x2x2x2", 2000, "fp32", "device", dt=0.5, M=4, graph=True)),
        # four three-level transmons, a gate on the sixteen subspace columns with a leakage penalty
        ("transmons_d81_fp32", _case("transmons", "3x3x3x3", 1000, "fp32", "device", dt=0.5, M=8)),
        # a seven-qubit gate, all columns, FP32
        ("qubits_d128_fp32", _case("qubits", "2x2x2x2x2x2x2", 500, "fp32", "device", dt=0.5, M=4)),
        # an eight-qubit gate, all columns, sixteen controls, the tensor-core form, at full length
        ("qubits_d256_bf16", _case("qubits", "2x2x2x2x2x2x2x2", 2000, "bf16", "device", dt=0.25, M=16)),
        # cat-state preparation in the lab frame, one trajectory of eight thousand slices
        ("cat_d154_fp32", _case("lab", "7x22", 8000, "fp32", "device", dt=0.005)),
        # the same system made robust: sixteen members, the series applied to the propagated columns
        ("cat_d154_E16_state_fp32", _case("lab", "7x22", 1000, "fp32", "device", dt=0.005, E=16,
                                          propagation="state", exponential="chebyshev")),
        # a sweep over sixteen problems of uneven size, one graph launch for all of them
        ("batch16_fp32", _case("mixed", "-", 4000, "fp32", "batch", dt=0.5, M=8, count=16)),
    ]
    return [dict(c, name=name) for name, c in named]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above: the same systems at other sizes, lengths and members."""
    qubits = lambda n: "x".join(["2"] * n)
    kind = rng.choice(["zz", "coupled", "autograd", "cavity", "transmons", "small_gate", "gate", "gate_bf16", "lab",
                       "lab_state", "batch"])
    if kind == "zz":
        return _case("zz", qubits(rng.randint(2, 4)), _log(rng, 50, 600), "fp64", "host", dt=0.5, M=4)
    if kind == "coupled":
        a, b = rng.randint(3, 6), rng.randint(3, 6)
        return _case("coupled", "%dx%d" % (a, b), _log(rng, 100, 500), "fp64", "host", dt=0.04, M=5)
    if kind == "autograd":
        return _case("qubits", qubits(rng.randint(2, 5)), _log(rng, 200, 4000), "fp32", "autograd", dt=0.5, M=4)
    if kind == "cavity":
        return _case("cavity", "%dx%d" % (rng.randint(3, 5), rng.randint(5, 12)), _log(rng, 300, 4000), "fp32",
                     "device", dt=1.0, graph=True)
    if kind == "transmons":
        dims, top = rng.choice([("3x3", 3000), ("3x3x3", 2000), ("4x4", 3000), ("3x4x3", 1500), ("4x4x4", 1000),
                                ("3x3x3x3", 1000), ("3x5x5", 1000)])
        E = rng.randint(1, 6)
        return _case("transmons", dims, max(100, _log(rng, 100, top) // E), "fp32", "device", dt=0.5,
                     M=2 * len(dims.split("x")), E=E)
    if kind == "small_gate":
        return _case("qubits", qubits(rng.randint(3, 6)), _log(rng, 200, 3000), "fp32", "device", dt=0.5, M=4,
                     graph=True)
    if kind == "gate":
        n = rng.randint(7, 8)
        return _case("qubits", qubits(n), _log(rng, 60, 2000 if n == 7 else 400), "fp32", "device",
                     dt=0.5 if n == 7 else 0.25, M=4)
    if kind == "gate_bf16":
        n = rng.randint(7, 8)
        return _case("qubits", qubits(n), _log(rng, 60, 2000), "bf16", "device", dt=0.5 if n == 7 else 0.25,
                     M=2 * rng.randint(2, n))
    if kind == "lab":
        return _case("lab", "%dx%d" % (rng.randint(4, 7), rng.randint(18, 22)), _log(rng, 300, 8000), "fp32",
                     "device", dt=0.005)
    if kind == "lab_state":
        exponential = rng.choice(["chebyshev", "chebyshev", "taylor"])
        return _case("lab", "%dx%d" % (rng.randint(4, 7), rng.randint(18, 22)),
                     _log(rng, 60, 1000 if exponential == "chebyshev" else 250), "fp32", "device", dt=0.005,
                     E=_log(rng, 1, 16), propagation="state", exponential=exponential)
    return _case("mixed", "-", _log(rng, 400, 4000), "fp32", "batch", dt=0.5, M=8, count=rng.randint(2, 12))


# ------------------------------------------------------------------------------------------
# the systems (hbar = 1, energies in rad/ns, time in ns)
# ------------------------------------------------------------------------------------------
SX = np.array([[0, 1], [1, 0]], np.complex128)
SY = np.array([[0, -1j], [1j, 0]], np.complex128)
SZ = np.array([[1, 0], [0, -1]], np.complex128)


def _lower(n):
    return np.diag(np.sqrt(np.arange(1.0, n)), 1).astype(np.complex128)


def _num(n):
    return np.diag(np.arange(float(n))).astype(np.complex128)


def _on(op, site, dims):
    out = np.ones((1, 1), np.complex128)
    for i, n in enumerate(dims):
        out = np.kron(out, op if i == site else np.eye(n))
    return out


def _haar(n, rng):
    q, r = np.linalg.qr(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))
    return q * (np.diag(r) / np.abs(np.diag(r)))[None, :]


def _gue(n, rng, norm):
    g = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    h = 0.5 * (g + g.conj().T)
    return h * (norm / np.max(np.abs(np.linalg.eigvalsh(h))))


def _paulis(dims, M):
    return np.stack([_on(op, q, dims) for q in range(len(dims)) for op in (SX, SY)][:M])


def _ladders(dims, sites, M):
    out = []
    for s in sites:
        b = _lower(dims[s])
        out += [_on(b + b.conj().T, s, dims), _on(1j * (b.conj().T - b), s, dims)]
    return np.stack(out[:M])


class _Problem:
    """One control problem in numpy: H_j = H0 + sum_k u[k, j] Hk[k] + delta_e Hdet."""

    def __init__(self, H0, Hk, dt, N, psi0, psiT, u, forbidden=(), weight=None, alpha=(1.0, 0, 0, 0, 0), delta=None,
                 Hdet=None):
        self.H0, self.Hk, self.dt, self.N, self.psi0, self.psiT = H0, Hk, dt, N, psi0, psiT
        self.forbidden = np.asarray(forbidden, np.int32)
        self.col_weight = np.ones(psi0.shape[1]) if weight is None else weight
        self.alpha = np.asarray(alpha, np.float64)
        self.u = u
        self.psiT_path = None
        self.delta = np.zeros(1) if delta is None else delta
        self.Hdet = Hdet


def _basis(d, k):
    v = np.zeros((d, 1), np.complex128)
    v[k, 0] = 1.0
    return v


def _problem(case, seed, index=0):
    rng = np.random.default_rng([int(seed), index])
    system, N, M, E, dt = case["system"], case["N"], case["M"], case["E"], case["dt"]
    if system == "mixed":      # one problem of a batch: uneven dimension, length and control count
        fixed = np.random.default_rng([7, case["count"], N, index])   # sizes belong to the case, not to the seed
        d = int(fixed.choice([4, 8, 16, 40, 81, 128]))
        N = int(fixed.integers(max(50, N // 20), N + 1))
        M = int(fixed.integers(2, 9))
        dims = {40: [4, 10], 81: [3, 3, 3, 3]}.get(d) or [2] * int(round(math.log2(d)))
        M = min(M, 2 * len(dims))
        Hk = _paulis(dims, M) if dims[0] == 2 else _ladders(dims, range(len(dims)), M)
        u = rng.normal(0.0, TWO_PI * 0.02, (M, N))
        return _Problem(_gue(d, rng, TWO_PI * 0.05), Hk, dt, N, np.eye(d, dtype=np.complex128), _haar(d, rng), u)
    dims = [int(x) for x in case["dims"].split("x")]
    d = int(np.prod(dims))
    delta = rng.normal(0.0, TWO_PI * 0.001, E) if E > 1 else None
    digits = np.array(np.unravel_index(np.arange(d), dims)).T
    if system == "zz":         # coupled qubits, a CNOT on the first two, the whole unitary
        H0 = sum(TWO_PI * 0.01 * _on(SZ, q, dims) @ _on(SZ, q + 1, dims) for q in range(len(dims) - 1))
        cnot = np.kron(np.array([[1, 0, 0, 0], [0, 1, 0, 0], [0, 0, 0, 1], [0, 0, 1, 0]], np.complex128),
                       np.eye(d // 4))
        u = rng.normal(0.0, TWO_PI * 0.02, (M, N))
        return _Problem(H0, _paulis(dims, M), dt, N, np.eye(d, dtype=np.complex128), cnot, u)
    if system == "coupled":    # two transmons in a rotating frame, a CNOT on the computational states
        al, J, det = -TWO_PI * 0.225, TWO_PI * 0.1, TWO_PI * 0.4
        H0 = det * _on(_num(dims[1]), 1, dims)
        for i, n in enumerate(dims):
            H0 = H0 + _on(0.5 * al * _num(n) @ (_num(n) - np.eye(n)), i, dims)
        hop = np.kron(_lower(dims[0]).conj().T, _lower(dims[1]))
        H0 = H0 + J * (hop + hop.conj().T)
        Hk = np.concatenate([_ladders(dims, [0, 1], 4), _on(_num(dims[1]), 1, dims)[None]])[:M]
        comp = [dims[1] * a + b for a in (0, 1) for b in (0, 1)]
        psi0, psiT = np.zeros((d, 4), np.complex128), np.zeros((d, 4), np.complex128)
        for s, k in enumerate(comp):
            psi0[k, s] = 1.0
            psiT[comp[(0, 1, 3, 2)[s]], s] = 1.0
        forb = np.where(np.any(digits >= 3, axis=1))[0]
        u = rng.normal(0.0, TWO_PI * 0.01, (M, N))
        return _Problem(H0, Hk, dt, N, psi0, psiT, u, forb, alpha=(1.0, 1e-6, 1e-4, 0.1 / (4 * N), 0.0))
    if system == "qubits":     # a random drift, Pauli controls, a random gate, the whole unitary
        u = rng.normal(0.0, TWO_PI * 0.02, (M, N))
        return _Problem(_gue(d, rng, TWO_PI * 0.05), _paulis(dims, M), dt, N, np.eye(d, dtype=np.complex128),
                        _haar(d, rng), u)
    if system == "cavity":     # a transmon and a cavity, dispersive, |g,0> -> |g,1>, top levels forbidden
        nt, nc = dims
        H0 = (0.5 * -TWO_PI * 0.225 * np.kron(_num(nt) @ (_num(nt) - np.eye(nt)), np.eye(nc))
              - TWO_PI * 0.002 * np.kron(_num(nt), _num(nc)))
        forb = np.where((digits[:, 0] == nt - 1) | (digits[:, 1] == nc - 1))[0]
        u = rng.normal(0.0, TWO_PI * 0.02, (M, N))
        return _Problem(H0, _ladders(dims, [0], M), dt, N, _basis(d, 0), _basis(d, 1), u, forb,
                        alpha=(1.0, 0, 0, 1.0 / N, 0))
    if system == "transmons":  # a transmon chain: a random gate on the qubit subspace, leakage forbidden
        H0 = np.zeros((d, d), np.complex128)
        for i, n in enumerate(dims):
            H0 += _on(-0.5 * TWO_PI * 0.2 * _num(n) @ (_num(n) - np.eye(n)), i, dims)
        for i in range(len(dims) - 1):
            hop = _on(_lower(dims[i]).conj().T, i, dims) @ _on(_lower(dims[i + 1]), i + 1, dims)
            H0 += TWO_PI * 0.005 * (hop + hop.conj().T)
        sub = np.where(np.all(digits <= 1, axis=1))[0]
        forb = np.where(np.any(digits >= 2, axis=1))[0]
        psiT, w = np.zeros((d, d), np.complex128), np.zeros(d)
        psiT[np.ix_(sub, sub)] = _haar(len(sub), rng)
        w[sub] = 1.0
        u = rng.normal(0.0, TWO_PI * 0.03, (M, N))
        Hdet = sum(_on(_num(n), i, dims) for i, n in enumerate(dims))
        return _Problem(H0, _ladders(dims, range(len(dims)), M), dt, N, np.eye(d, dtype=np.complex128), psiT, u, forb,
                        w, (1.0, 0, 0, 1.0 / (len(sub) * N), 0), delta, Hdet)
    nq, nr = dims              # "lab": a transmon and a cavity in the lab frame, vacuum -> cat state
    b, a = _lower(nq), _lower(nr)
    H0 = (np.kron(TWO_PI * 3.5 * _num(nq) - 0.5 * TWO_PI * 0.225 * _num(nq) @ (_num(nq) - np.eye(nq)), np.eye(nr))
          + np.kron(np.eye(nq), TWO_PI * 3.9 * _num(nr))
          + TWO_PI * 0.1 * np.kron(b + b.conj().T, a + a.conj().T))
    nb = np.kron(_num(nq), np.eye(nr)).astype(np.complex128)
    Hk = np.stack([np.kron(b + b.conj().T, np.eye(nr)), nb]).astype(np.complex128)
    coherent = lambda z: np.array([z ** k / math.sqrt(math.factorial(k)) for k in range(nr)])
    cat = coherent(2.0) + coherent(-2.0)
    psiT = np.zeros((d, 1), np.complex128)
    psiT[:nr, 0] = cat / np.linalg.norm(cat)
    forb = np.where((digits[:, 0] >= 3) | (digits[:, 1] >= nr - 2))[0]
    u = rng.normal(0.0, TWO_PI * 0.02, (M, N))
    return _Problem(H0, Hk, dt, N, _basis(d, 0), psiT, u, forb, alpha=(1.0, 0, 1e-4, 1.0 / N, 0), delta=delta, Hdet=nb)


def _problems(case, seed):
    pbs = [_problem(case, seed, i) for i in range(case["count"])]
    if case["precision"] != "fp64":     # float32 parameters
        for pb in pbs:
            pb.u = pb.u.astype(np.float32).astype(np.float64)
    return pbs


# ------------------------------------------------------------------------------------------
# one pass
# ------------------------------------------------------------------------------------------
_stream = None


def _program_stream():
    """The stream that the program runs on: one for all of its contexts (a graph is not captured
    from the default stream)."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


class _State:
    pass


def prepare(case, seed):
    pbs = _problems(case, seed)
    s = _State()
    s.entry, s.stream = case["entry"], _program_stream()
    own = s.entry in ("host", "batch")
    s.ctxs = []
    for pb in pbs:
        c = qoc.Context(case["precision"], graph=case["graph"], propagation=case["propagation"],
                        exponential=case["exponential"], stream=None if own else s.stream.cuda_stream)
        c.set_problem(pb)
        s.ctxs.append(c)
    if s.entry == "host":
        s.u = pbs[0].u
        return s
    sizes = [pb.u.size for pb in pbs]
    flat = torch.from_numpy(np.concatenate([pb.u.ravel() for pb in pbs]).astype(np.float32)).cuda()
    s.shape = pbs[0].u.shape
    if s.entry == "autograd":
        s.u = flat.reshape(s.shape).requires_grad_(True)
        torch.cuda.synchronize()
        return s
    s.u32, s.u = flat, flat.double()
    s.grad = torch.zeros_like(s.u)
    s.out = torch.zeros(len(pbs), 6, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    if s.entry == "batch":
        at = [0] + list(np.cumsum(sizes))[:-1]
        s.batch = qoc.Batch(s.ctxs, [s.u.data_ptr() + 8 * int(a) for a in at],
                            [s.grad.data_ptr() + 8 * int(a) for a in at],
                            [s.out.data_ptr() + 48 * i for i in range(len(pbs))], s.stream.cuda_stream)
    return s


def run(state):
    s = state
    if s.entry == "host":
        cost, grad, terms = s.ctxs[0].evaluate(s.u)
        return {"cost": cost, "grad": grad, "terms": terms}
    with torch.cuda.stream(s.stream):
        if s.entry == "autograd":
            s.u.grad = None
            cost, terms = qoc.cost(s.ctxs[0], s.u.double())
            loss = cost.float()
            loss.backward()
            return {"cost": loss.detach(), "terms": terms.detach().float(), "grad": s.u.grad}
        s.u.copy_(s.u32)
        if s.entry == "batch":
            s.batch.launch(s.stream.cuda_stream)
            return {"out": s.out.float(), "grad": s.grad.float()}
        s.ctxs[0].evaluate_device(s.u.data_ptr(), s.grad.data_ptr(), s.out.data_ptr())
        return {"out": s.out[0].float(), "grad": s.grad.reshape(s.shape).float()}


# ------------------------------------------------------------------------------------------
# what a pass cannot do without
# ------------------------------------------------------------------------------------------
def _theta(pb):
    one = lambda a: float(np.max(np.sum(np.abs(a), axis=0)))
    t = one(pb.H0) + np.max(np.sum(np.abs(pb.u) * np.array([one(h) for h in pb.Hk])[:, None], axis=0))
    return pb.dt * (t + (float(np.max(np.abs(pb.delta))) * one(pb.Hdet) if len(pb.delta) > 1 else 0.0))


def work(case):
    """bytes: the Hamiltonians, the states and the controls in, the gradient out.  flops: the cheaper
    of two ways to do one slice and member: the exponential as a polynomial of degree about
    theta + 8 by matrix products (2 sqrt(degree) of them, twice that for its reverse mode) with one
    product by the columns each way, or the polynomial applied to the columns (forward, backward and
    the reverse mode's recomputation and rank-one updates); and M contractions with the controls."""
    total = {"bytes": 0.0, "flops": 0.0}
    for pb in _problems(case, 1):
        d, M, S, E, N = pb.H0.shape[0], pb.Hk.shape[0], int(np.sum(pb.col_weight > 0)), len(pb.delta), pb.N
        wide = 16 if case["precision"] == "fp64" else 8
        degree = _theta(pb) + (20 if wide == 16 else 8)
        products = 3 * 2 * math.sqrt(degree) * 8.0 * d ** 3 + 3 * 8.0 * d * d * S
        columns = 5 * degree * 8.0 * d * d * S
        sparse = max(1.0, float(np.mean([np.count_nonzero(h) for h in pb.Hk])))   # a control's non-zero entries
        total["flops"] += E * N * (min(products, columns) + 4.0 * M * sparse)
        total["bytes"] += wide * ((M + 2) * d * d + 2 * d * S) + wide * M * N
    return total


# ------------------------------------------------------------------------------------------
# the same evaluation in 64 bits
# ------------------------------------------------------------------------------------------
_DEGREE = 18     # Taylor at a norm of at most 1: remainder below 1e-17


def _expm(X, n):
    """exp(X) by Taylor (Paterson-Stockmeyer, blocks of four) at X / 2^n and n squarings."""
    X = X / 2.0 ** n
    c = [1.0 / math.factorial(k) for k in range(_DEGREE + 1)]
    eye = torch.eye(X.shape[-1], dtype=X.dtype, device=X.device)
    X2 = X @ X
    X3 = X2 @ X
    X4 = X2 @ X2
    W = c[16] * eye + c[17] * X + c[18] * X2
    for q in (12, 8, 4, 0):
        W = X4 @ W + (c[q] * eye + c[q + 1] * X + c[q + 2] * X2 + c[q + 3] * X3)
    for _ in range(n):
        W = W @ W
    return W


def _apply(X, v, n):
    """exp(X) v by the same series, without forming exp(X)."""
    X = X / 2.0 ** n
    for _ in range(2 ** n):
        z = v
        for k in range(_DEGREE, 0, -1):
            z = v + (X @ z) / k
        v = z
    return v


def _exact_one(pb):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    z = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.complex128)).to(dev)
    cols = np.where(pb.col_weight > 0)[0]
    H0, Hk, psi0, psiT = z(pb.H0), z(pb.Hk), z(pb.psi0[:, cols]), z(pb.psiT[:, cols])
    u = torch.from_numpy(pb.u).to(dev)
    w = torch.from_numpy(pb.col_weight[cols]).to(dev)
    M, N = pb.u.shape
    d, S, E = H0.shape[0], len(cols), len(pb.delta)
    n = max(0, math.ceil(math.log2(max(_theta(pb), 1e-9))))
    F = torch.from_numpy(pb.forbidden.astype(np.int64)).to(dev)
    a_fid, a_amp, a_var, a_forb, a_time = (float(x) for x in pb.alpha)
    W = w.sum()
    grad = torch.zeros(M, N, dtype=torch.float64, device=dev)
    fid = forb = time = 0.0
    by_columns = 2 ** n * _DEGREE * S < (7 + n) * d
    chunk = max(1, int(1.5e7 // (d * d)))

    def X_of(j0, j1, e):
        H = H0 + torch.einsum("kj,kab->jab", u[:, j0:j1].to(H0.dtype), Hk)
        if pb.Hdet is not None and pb.delta[e] != 0.0:
            H = H + float(pb.delta[e]) * z(pb.Hdet)
        return -1j * pb.dt * H

    U = torch.empty(N, d, d, dtype=H0.dtype, device=dev)
    psi = torch.empty(N + 1, d, S, dtype=H0.dtype, device=dev)
    G = torch.empty(N + 1, d, S, dtype=H0.dtype, device=dev)
    for e in range(E):
        for j0 in range(0, N, chunk):
            U[j0:j0 + chunk] = _expm(X_of(j0, min(N, j0 + chunk), e), n)
        psi[0] = psi0
        for j in range(N):
            torch.matmul(U[j], psi[j], out=psi[j + 1])
        over = torch.einsum("as,jas,s->j", psiT.conj(), psi[1:], w.to(H0.dtype)) / W
        fid += float(1.0 - over[-1].abs() ** 2) / E
        if len(F):
            forb += float((psi[1:, F, :].abs() ** 2 * w).sum()) / E
        time += float(1.0 - (over.abs() ** 2).mean()) / E
        G.zero_()                                     # the sources, then the costates on top of them
        if len(F) and a_forb:
            G[1:, F, :] = (2.0 * a_forb / E) * psi[1:, F, :] * w
        if a_time:
            G[1:] += (-2.0 * a_time / (N * E)) * over[:, None, None] * psiT * (w / W)
        G[N] += (-2.0 * a_fid / E) * over[-1] * psiT * (w / W)
        for j in range(N - 1, 0, -1):
            G[j].addmm_(U[j].mH, G[j + 1])
        for j0 in range(0, N, chunk):
            j1 = min(N, j0 + chunk)
            X = X_of(j0, j1, e).requires_grad_(True)
            g, p = G[j0 + 1:j1 + 1], psi[j0:j1]
            if by_columns:
                Xbar, = torch.autograd.grad(_apply(X, p, n), X, g)
            else:
                Xbar, = torch.autograd.grad(_expm(X, n), X, g @ p.mH)
            grad[:, j0:j1] += torch.einsum("jab,kab->kj", Xbar.conj(), -1j * pb.dt * Hk).real
    grad += 2.0 * a_amp * u
    du = u[:, 1:] - u[:, :-1]
    grad[:, 1:] += 2.0 * a_var * du
    grad[:, :-1] -= 2.0 * a_var * du
    terms = [fid, float((u * u).sum()), float((du * du).sum()), forb, time]
    total = sum(a * t for a, t in zip((a_fid, a_amp, a_var, a_forb, a_time), terms))
    return total, np.array(terms), grad.cpu().numpy()


def exact(case, seed):
    got = [_exact_one(pb) for pb in _problems(case, seed)]
    cost, terms, grad = got[0]
    if case["entry"] in ("host", "autograd"):
        return {"cost": cost, "terms": terms, "grad": grad}
    outs = np.stack([np.concatenate([[c], t]) for c, t, _ in got])
    if case["entry"] == "batch":
        return {"out": outs, "grad": np.concatenate([g.ravel() for _, _, g in got])}
    return {"out": outs[0], "grad": grad}
