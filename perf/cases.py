"""Performance cases: the evaluations a robust-GRAPE program asks of this library.

A case is one call as an optimiser, a validation run, a serving loop or a host
without ``cudaMalloc`` makes it: the controls of this iterate go in, F (with
dF/du, or |O|^2 per trajectory) comes out.  Shapes follow the repository's
workloads (parallel X and CNOT on 8 to 50 qubits, GHZ on 30, the echo whose
bonds reach the cap, the gate objective in operator form, the serving mix);
ensembles are cut so that one pass takes well under two seconds.

Controls are what the path meets in earnest: random starts on short chains,
and on long chains iterates near a solution (an exact pulse of the target at
zero crosstalk plus jitter) or an echo (random controls, then their time
reverse negated: the entanglement of random controls with a final overlap of
order one).  With random controls on a long chain every overlap is near 1e-10
and its digits say nothing about the arithmetic; these keep it well above.

``run`` returns every output whole.  ``exact`` evaluates the same Trotterised
circuit on dense state vectors in torch (autograd for the gradient) wherever
the case truncates nothing but numerical zeros and the vectors are small.
"""
import functools
import math

import numpy as np
import torch

from paper_2603_03639_gb300 import autotune
from paper_2603_03639_gb300.autograd import fidelity
from paper_2603_03639_gb300.tnrc import Context, fidelity_static

BASE = {"call": "grad", "N": 8, "K": 20, "dt": 0.05, "chi": 16, "M": 16, "P": 4, "C": 2, "g": "none",
        "pulse": "random", "sigma": 0.5, "target": "x", "dist": 0, "scale": 0.05, "terms": 1, "order": 2,
        "substeps": 1, "operator": False, "bond": 8}


def _case(name=None, **kw):
    c = dict(BASE, **kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a host that may not allocate device memory asks for one small fidelity
        _case("static_x6", call="static", N=6, K=6, chi=8, M=4, P=2, bond=4),
        # an optimiser's first iterations on the small parallel-X problem
        _case("grad_x8", bond=12),
        # the gate objective of a short chain: first-order slices, the paper's first-stage ensemble of 6 (N - 1)
        _case("grad_gate4", N=4, K=10, dt=0.1, chi=16, M=18, P=1, C=3, g="all", pulse="near", operator=True,
              order=1, terms=3, scale=0.3, bond=8),
        # the same problem class driven from torch: forward and backward of the autograd function
        _case("autograd_cnot12", call="autograd", N=12, K=24, chi=64, M=24, P=4, C=3, g="pairs", pulse="near",
              target="cnot", dist=1, bond=8),
        # the serving loop's launch form (own stream, pooled, captured graph) on a Heisenberg-target request
        _case("served_heis10", call="served", N=10, K=30, dt=0.1, chi=32, M=24, P=1, C=3, g="all", sigma=1.5,
              target="heis", terms=3, bond=18),
        # an odd chain, odd ensemble, several Trotter steps per bin
        _case("grad_x13_substeps", N=13, K=11, dt=0.15, chi=32, M=37, P=3, pulse="echo", target="input", substeps=3,
              bond=9),
        # parallel X on 50 qubits near the solution
        _case("grad_x50", N=50, K=64, chi=32, M=64, P=8, pulse="near", scale=0.1, bond=6),
        # validation of a pulse on fresh samples: fidelities only
        _case("fid_x50", call="fidelity", N=50, K=64, chi=32, M=160, P=4, pulse="near", scale=0.1, bond=6),
        # parallel CNOT on 50 qubits (the benchmark's shape) near the solution
        _case("grad_cnot50", N=50, K=100, chi=64, M=38, P=8, C=3, g="pairs", pulse="near", target="cnot", dist=1,
              bond=8),
        # GHZ preparation on 30 qubits with the entanglement of random controls
        _case("grad_ghz30", N=30, K=64, chi=64, M=152, P=1, C=3, g="all", pulse="echo", target="ghz", bond=10),
        # bonds at the cap: strong controls on 12 qubits, theta up to 64 x 64
        _case("grad_echo12_cap", N=12, K=8, dt=0.5, chi=32, M=76, P=1, C=3, g="all", pulse="echo", sigma=1.5,
              target="input", scale=0.1, bond=24),
        # the gate objective on a long chain, operator bonds at D_max = 20
        _case("grad_gate24", N=24, K=24, chi=20, M=38, P=1, C=3, g="pairs", pulse="near", target="cnot", dist=1,
              operator=True, bond=14),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["static", "small", "gate", "autograd", "served", "odd", "xlong", "fidlong", "cnotlong",
                       "ghzlong", "cap", "gatelong"])
    if kind == "static":
        return _case(call="static", N=rng.randint(2, 8), K=_log(rng, 2, 12), chi=8, M=_log(rng, 1, 12),
                     P=rng.randint(1, 3), bond=4)
    if kind == "small":
        return _case(N=rng.randint(3, 9), K=_log(rng, 4, 40), chi=rng.choice([16, 32, 64]), M=_log(rng, 2, 64),
                     P=rng.randint(1, 5), order=rng.choice([1, 2]), bond=10)
    if kind == "gate":
        return _case(N=rng.randint(2, 5), K=_log(rng, 4, 20), dt=0.1, chi=16, M=_log(rng, 6, 48), P=1, C=3, g="all",
                     pulse="near", operator=True, order=rng.choice([1, 2]), terms=rng.choice([1, 3]), scale=0.2,
                     bond=8)
    if kind == "autograd":
        return _case(call="autograd", N=2 * rng.randint(3, 7), K=_log(rng, 8, 32), chi=64, M=_log(rng, 4, 40),
                     P=rng.randint(1, 5), C=3, g="pairs", pulse="near", target="cnot", dist=1, bond=8)
    if kind == "served":
        return _case(call="served", N=rng.choice([8, 9, 10]), K=_log(rng, 10, 30), dt=0.1, chi=rng.choice([20, 32]),
                     M=_log(rng, 4, 24), P=1, C=3, g="all", sigma=1.5, target="heis", terms=rng.choice([1, 3]),
                     bond=18)
    if kind == "odd":
        return _case(N=rng.choice([5, 7, 9, 11, 13, 15]), K=rng.randint(3, 12), dt=0.15, chi=32, M=_log(rng, 3, 45),
                     P=rng.randint(1, 4), pulse="echo", target="input", substeps=rng.randint(1, 3),
                     order=rng.choice([1, 2]), bond=9)
    if kind == "xlong":
        return _case(N=rng.randint(20, 50), K=_log(rng, 16, 64), chi=32, M=_log(rng, 8, 64), P=rng.randint(2, 8),
                     pulse="near", scale=0.1, bond=6)
    if kind == "fidlong":
        return _case(call="fidelity", N=rng.randint(20, 50), K=_log(rng, 16, 64), chi=32, M=_log(rng, 20, 160),
                     P=rng.randint(1, 4), pulse="near", scale=0.1, bond=6)
    if kind == "cnotlong":
        return _case(N=2 * rng.randint(10, 25), K=_log(rng, 24, 100), chi=64, M=_log(rng, 4, 38), P=rng.randint(2, 8),
                     C=3, g="pairs", pulse="near", target="cnot", dist=1, bond=8)
    if kind == "ghzlong":
        return _case(N=rng.randint(16, 30), K=2 * _log(rng, 8, 32), chi=64, M=_log(rng, 16, 152), P=1, C=3, g="all",
                     pulse="echo", target="ghz", bond=10)
    if kind == "cap":
        return _case(N=rng.randint(9, 12), K=2 * rng.randint(2, 4), dt=0.5, chi=rng.choice([12, 16, 24, 32]),
                     M=_log(rng, 8, 76), P=1, C=3, g="all", pulse="echo", sigma=1.5, target="input", scale=0.1,
                     bond=24)
    return _case(N=2 * rng.randint(6, 12), K=_log(rng, 8, 24), chi=20, M=_log(rng, 8, 38), P=1, C=3, g="pairs",
                 pulse="near", target="cnot", dist=1, operator=True, bond=14)


# -- inputs ---------------------------------------------------------------------------------------------------------

def _pulse(c):
    """An exact pulse u[K][C][N] of the case's target at zero crosstalk."""
    K, N, dt = c["K"], c["N"], c["dt"]
    u = np.zeros((K, c["C"], N))
    if c["target"] == "x":
        u[:, 0, :] = math.pi / (2 * K * dt)
        return u
    # CNOT = e^{i pi/4 Z_c} e^{i pi/4 X_t} e^{-i pi/4 Z_c X_t}: the control's Z rotation from x, y, x pulses, the ZZ
    # coupling between two target y rotations, a target x rotation; six stretches of K // 6 slices
    n = K // 6
    if n < 1:
        raise ValueError("the CNOT pulse needs six slices")
    a = math.pi / 4 / (n * dt)
    ctl, tgt = slice(0, N, 2), slice(1, N, 2)
    s = [slice(i * n, (i + 1) * n) for i in range(6)]
    u[s[0], 0, ctl] = -a
    u[s[0], 1, tgt] = -a
    u[s[1], 1, ctl] = -a
    u[s[2], 0, ctl] = a
    u[s[3], 2, ctl] = a
    u[s[4], 1, tgt] = a
    u[s[5], 0, tgt] = -a
    return u


def _controls(c, rng):
    K, C, N = c["K"], c["C"], c["N"]
    if c["pulse"] == "random":
        return rng.normal(0.0, c["sigma"], size=(K, C, N))
    if c["pulse"] == "near":
        return _pulse(c) + rng.normal(0.0, 0.05, size=(K, C, N))
    h = rng.normal(0.0, c["sigma"], size=(K // 2, C, N))
    mid = rng.normal(0.0, 0.05, size=(K % 2, C, N))
    return np.concatenate([h, mid, -h[::-1]])


def _mask(c):
    m = np.ones((c["C"], c["N"]), dtype=np.uint8)
    if c["C"] == 3:
        m[2] = 0
        m[2, 0:c["N"] - 1:2 if c["g"] == "pairs" else 1] = 1 if c["g"] != "none" else 0
    return m


def _splitmix(seed, i):
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + (i + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _noise(c, seed):
    """J[M][N-1] (or [M][N-1][3]) from the library's counter-based generator."""
    shape = (c["M"], c["N"] - 1) + ((3,) if c["terms"] == 3 else ())
    i = np.arange(int(np.prod(shape)), dtype=np.uint64)
    u = lambda k: (_splitmix(seed, k) >> np.uint64(11)).astype(np.float64)  # noqa: E731
    if c["dist"] == 0:
        return (c["scale"] * (2 * u(i) * 2.0 ** -53 - 1)).reshape(shape)
    r = np.sqrt(-2 * np.log((u(2 * i) + 1) * 2.0 ** -53))
    return (c["scale"] * r * np.cos(2 * np.pi * u(2 * i + np.uint64(1)) * 2.0 ** -53)).reshape(shape)


@functools.lru_cache(maxsize=None)
def _heisenberg(N, chi):
    """Ground state of sum_j XX + YY + ZZ on an open chain, cut into an MPS."""
    dim = 1 << N
    idx = np.arange(dim)
    h = np.zeros((dim, dim))
    for b in range(N - 1):
        anti = ((idx >> (N - 1 - b)) ^ (idx >> (N - 2 - b))) & 1 == 1
        h[idx, idx] += np.where(anti, -1.0, 1.0)
        h[idx[anti], idx[anti] ^ (3 << (N - 2 - b))] += 2.0
    # a small field splits the doublet of an odd chain
    h[idx, idx] += 1e-3 * sum(1.0 - 2 * ((idx >> j) & 1) for j in range(N)) if N % 2 else 0.0
    psi = np.linalg.eigh(h)[1][:, 0].astype(np.complex128)
    sites, rest, dl = [], psi.reshape(1, dim), 1
    for _ in range(N - 1):
        w, s, vh = np.linalg.svd(rest.reshape(dl * 2, -1), full_matrices=False)
        k = max(1, min(chi, int(np.count_nonzero(s > 1e-12 * s[0]))))
        sites.append(w[:, :k].reshape(dl, 2, k))
        rest = s[:k, None] * vh[:k] / np.linalg.norm(s[:k])
        dl = k
    return sites + [rest.reshape(dl, 2, 1)]


def _cnot_sites(c, t, flip):
    a = np.zeros((1, c[0].size, 2), dtype=np.complex128)
    a[0, :, 0], a[0, :, 1] = c
    return [a, np.stack([t, flip]).reshape(2, -1, 1)]


def _states(c, rng):
    """(inputs, targets): lists of P lists of site tensors (D, d, D')."""
    N, P = c["N"], c["P"]
    prod = lambda vs: [np.asarray(v, dtype=np.complex128).reshape(1, -1, 1) for v in vs]  # noqa: E731
    if c["operator"]:
        eye, x = np.eye(2).ravel() / math.sqrt(2), np.array([0, 1, 1, 0]) / math.sqrt(2)
        if c["target"] == "x":
            tgt = prod([x] * N)
        else:
            p0, p1 = np.array([1, 0, 0, 0]) / math.sqrt(2), np.array([0, 0, 0, 1]) / math.sqrt(2)
            tgt = sum((_cnot_sites((p0, p1), eye + 0j, x + 0j) for _ in range(N // 2)), [])
        return [prod([eye] * N)] * P, [tgt] * P
    if c["target"] in ("ghz", "heis"):
        zero = prod([[1, 0]] * N)
        if c["target"] == "heis":
            return [zero] * P, [_heisenberg(N, c["chi"])] * P
        d = np.zeros((2, 2, 2), dtype=np.complex128)
        d[0, 0, 0] = d[1, 1, 1] = 1
        first = (np.eye(2) / math.sqrt(2) + 0j).reshape(1, 2, 2)
        return [zero] * P, [[first] + [d] * (N - 2) + [np.eye(2, dtype=np.complex128).reshape(2, 2, 1)]] * P
    ins, tgs = [], []
    for _ in range(P):
        z = rng.normal(size=(N, 2)) + 1j * rng.normal(size=(N, 2))
        z /= np.linalg.norm(z, axis=1, keepdims=True)
        ins.append(prod(z))
        if c["target"] == "input":
            tgs.append(prod(z))
        elif c["target"] == "x":
            tgs.append(prod(z[:, ::-1]))
        else:
            tgs.append(sum((_cnot_sites((np.array([z[i, 0], 0]), np.array([0, z[i, 1]])), z[i + 1], z[i + 1, ::-1])
                            for i in range(0, N, 2)), []))
    return ins, tgs


def _pack(sites):
    dims = np.array([1] + [s.shape[2] for s in sites], dtype=np.int32)
    return dims, np.concatenate([np.ascontiguousarray(s, dtype=np.complex128).ravel() for s in sites])


def _inputs(c, seed):
    rng = np.random.default_rng(seed)
    u = _controls(c, rng)
    ins, tgs = _states(c, rng)
    return u, _noise(c, seed), ins, tgs


# -- the library's side -----------------------------------------------------------------------------------------------

class _State:
    pass


def prepare(case, seed):
    c = case
    u, J, ins, tgs = _inputs(c, seed)
    s = _State()
    s.c, s.u, s.J = c, np.ascontiguousarray(u), np.ascontiguousarray(J)
    s.ins, s.tgs, s.mask = [_pack(m) for m in ins], [_pack(m) for m in tgs], _mask(c)
    s.form = dict(crosstalk=c["terms"], order=c["order"], substeps=c["substeps"], operator=c["operator"])
    if c["call"] == "static":
        return s
    shape = (c["N"], c["K"], c["chi"], c["M"], c["P"], c["C"])
    stream = None
    warps = ctas = 0
    if c["call"] == "served":
        s.side = torch.cuda.Stream()
        stream = s.side.cuda_stream
    else:   # the launch shape the library's tuner has cached for this problem, as bench.py takes it
        warps, ctas = autotune.lookup(*shape, grad=c["call"] != "fidelity", operator=c["operator"])
    s.ctx = Context(c["N"], c["K"], c["dt"], c["chi"], c["M"], c["C"], s.ins, s.tgs, mask=s.mask, stream=stream,
                    warps=warps, ctas_per_sm=ctas, **s.form)
    if c["call"] != "served":
        s.ctx.set_svd_shape(autotune.lookup_pairs(*shape, grad=c["call"] != "fidelity", operator=c["operator"]))
    s.ctx.set_noise(s.J)
    if c["call"] in ("autograd", "served"):
        s.ud = torch.tensor(s.u, dtype=torch.float64, device="cuda", requires_grad=c["call"] == "autograd")
    if c["call"] == "served":
        s.ctx.set_pooled(True)
        s.ctx.set_graphs(True)
        s.F = torch.zeros(1, dtype=torch.float64, device="cuda")
        s.g = torch.zeros(s.u.shape, dtype=torch.float64, device="cuda")
    return s


def run(state):
    s, c = state, state.c
    if c["call"] == "static":
        F, pt = fidelity_static(c["N"], c["K"], c["dt"], c["chi"], c["C"], s.ins, s.tgs, s.u, s.J, mask=s.mask,
                                per_traj=True, **s.form)
        return {"F": F, "per_traj": pt}
    if c["call"] == "autograd":
        F = fidelity(s.ud, s.ctx)
        (g,) = torch.autograd.grad(F, s.ud)
        return {"F": F.detach(), "grad": g}
    if c["call"] == "served":
        s.ctx.set_controls_dev(s.ud.data_ptr())
        s.ctx.evaluate_dev(s.F.data_ptr(), s.g.data_ptr())
        s.ctx.sync()   # a server waits for the request before it answers
        return {"F": s.F, "grad": s.g}
    s.ctx.set_controls(s.u)
    if c["call"] == "fidelity":
        F, pt = s.ctx.fidelity(per_traj=True)
        return {"F": F, "per_traj": pt}
    F, g = s.ctx.fidelity_grad()
    return {"F": F, "grad": g}


def work(case):
    """Each input read and each output written once; the arithmetic of the truncated TEBD sweeps (complex, 8 flops a
    multiply-add) at the bond dimension that the case's states typically reach, an SVD counted as 22 n^3 complex
    multiply-adds' worth of flops (Golub and Van Loan's thin SVD on square n)."""
    c = case
    N, K, T = c["N"], c["K"], c["M"] * c["P"]
    d = 4 if c["operator"] else 2
    b = min(c["bond"], c["chi"], 2 ** (N // 2) if d == 2 else 4 ** (N // 2))
    grad = c["call"] in ("grad", "autograd", "served")
    layers = (2 * K * c["substeps"] + (1 if c["order"] == 2 else 0)) * (N - 1) / 2.0
    n = d * b
    update = 8.0 * n * n * b + 32.0 * n * n + 4 * 22.0 * n ** 3 + 8.0 * n * n * b
    env = 8.0 * 2 * 2 * 2 * d * b ** 3 + 8.0 * d * d * 3 * b ** 3
    flops = T * layers * (update + ((update + env) if grad else 0.0))
    dims = d * (4 if c["target"] in ("ghz", "cnot") else b * b if c["target"] == "heis" else 1) + d
    nbytes = 8.0 * (K * c["C"] * N * (2 if grad else 1) + c["M"] * (N - 1) * c["terms"] + 1 + T) + 16.0 * c["P"] * N * dims
    return {"bytes": nbytes, "flops": flops}


# -- 64-bit values ------------------------------------------------------------------------------------------------------

def _dense(sites):
    v = sites[0].reshape(sites[0].shape[1], -1)
    for s in sites[1:]:
        v = np.tensordot(v, s, axes=([v.ndim - 1], [0])).reshape(v.shape[0] * s.shape[1], -1)
    return v.reshape(-1)


def _kron(a, b):
    return torch.kron(a, b)


def exact(case, seed):
    """F and dF/du (or |O|^2) of the same Trotterised circuit on dense vectors; None where the bonds are cut at chi or
    the vectors are large."""
    c = case
    N, K, M, P, C = (c[k] for k in ("N", "K", "M", "P", "C"))
    d = 4 if c["operator"] else 2
    full = d ** (N // 2)
    if (c["operator"] and N > 5) or N > 13 or c["chi"] < full or M * P * d ** N * K * c["substeps"] * N > 3e9:
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    u0, J, ins, tgs = _inputs(c, seed)
    cx = dict(dtype=torch.complex128, device=dev)
    I2 = torch.eye(2, **cx)
    X = torch.tensor([[0, 1], [1, 0]], **cx)
    Y = torch.tensor([[0, -1j], [1j, 0]], **cx)
    Z = torch.tensor([[1, 0], [0, -1]], **cx)
    XI, YI, IX, IY = _kron(X, I2), _kron(Y, I2), _kron(I2, X), _kron(I2, Y)
    pair = [_kron(X, X), _kron(Y, Y), _kron(Z, Z)]
    grad = c["call"] in ("grad", "autograd", "served")
    u = torch.tensor(u0, dtype=torch.float64, device=dev, requires_grad=grad)
    um = u * torch.tensor(_mask(c), dtype=torch.float64, device=dev)
    Jt = torch.tensor(J, dtype=torch.float64, device=dev).reshape(M, N - 1, -1)
    dts = c["dt"] / c["substeps"]

    def inter(b):      # [M][K][4][4]
        h = 0
        for q in range(Jt.shape[2]):
            h = h + Jt[:, b, q].to(torch.complex128)[:, None, None, None] * pair[q - Jt.shape[2]]
        if C == 3:
            h = h + um[:, 2, b].to(torch.complex128)[None, :, None, None] * pair[2]
        return h.expand(M, K, 4, 4)

    def bond(b):
        w = lambda e: (0.5 if 0 < b + e < N - 1 else 1.0)  # noqa: E731
        t = lambda q, i, G: um[:, q, i].to(torch.complex128)[:, None, None] * G  # noqa: E731
        return inter(b) + (w(0) * (t(0, b, XI) + t(1, b, YI)) + w(1) * (t(0, b + 1, IX) + t(1, b + 1, IY)))[None]

    def two(psi, G, b):
        v = psi.reshape(M, -1, 4, 2 ** (N - 2 - b), psi.shape[-1])
        return torch.einsum("mij,majkr->maikr", G, v).reshape(psi.shape)

    def one(psi, G, i):   # G [2][2], the same for every sample
        v = psi.reshape(M, 2 ** i, 2, 2 ** (N - 1 - i), psi.shape[-1])
        return torch.einsum("ij,majkr->maikr", G, v).reshape(psi.shape)

    if c["operator"]:     # U acts on the columns of the identity; O = tr(U_T^dag U) / 2^N
        R = 2 ** N
        psi = torch.eye(R, **cx)[None].repeat(M, 1, 1)
        t4 = _dense(tgs[0]).reshape([2, 2] * N).transpose(list(range(0, 2 * N, 2)) + list(range(1, 2 * N, 2)))
        tg = torch.tensor(t4.reshape(R, R) * math.sqrt(2.0) ** N, **cx)
    else:
        psi = torch.tensor(np.stack([_dense(m) for m in ins], axis=-1), **cx)[None].repeat(M, 1, 1)
        psi = psi / torch.linalg.vector_norm(psi, dim=1, keepdim=True)
        tg = torch.tensor(np.stack([_dense(m) for m in tgs], axis=-1), **cx)
        tg = tg / torch.linalg.vector_norm(tg, dim=0, keepdim=True)
    if c["order"] == 2:
        half = {b: torch.linalg.matrix_exp(-0.5j * dts * bond(b)) for b in range(0, N - 1, 2)}
        whole = {b: torch.linalg.matrix_exp(-1j * dts * bond(b)) for b in range(1, N - 1, 2)}
    else:
        whole = {b: torch.linalg.matrix_exp(-1j * dts * inter(b)) for b in range(N - 1)}
        rot = [[torch.linalg.matrix_exp(-1j * dts * um[:, q, i].to(torch.complex128)[:, None, None] * G)
                for i in range(N)] for q, G in ((1, Y), (0, X))]
    for k in range(K):
        for _ in range(c["substeps"]):
            if c["order"] == 2:
                for part in (half, whole, half):
                    for b, G in part.items():
                        psi = two(psi, G[:, k], b)
            else:
                for b in list(range(1, N - 1, 2)) + list(range(0, N - 1, 2)):
                    psi = two(psi, whole[b][:, k], b)
                for q in rot:
                    for i in range(N):
                        psi = one(psi, q[i][k], i)
    O = torch.einsum("ir,mir->mr", tg.conj(), psi)
    if c["operator"]:
        O = O.sum(dim=1, keepdim=True) / 2 ** N
    p2 = O.real ** 2 + O.imag ** 2
    F = p2.mean()
    if not grad:
        return {"F": F, "per_traj": p2}
    (g,) = torch.autograd.grad(F, u)
    F = F.detach()
    return {"F": F.reshape(1) if c["call"] == "served" else F, "grad": g}
