"""Gradients where overlaps are small or tensors dense: the environments span many
decades, or their sums many terms, and the gradient is compared with the oracle's
relative to its own size."""
import numpy as np
import pytest

import synth
from oracle import robust
from tests._util import TOL_G_REL, gpu_context, grad_close, oracle_problem

pytestmark = pytest.mark.gpu


def _both(w, u, J, ins, tgs):
    mask = np.ones((w.C, w.N), dtype=np.uint8)
    Fo, go, Oo = robust.ensemble(oracle_problem(w, u, mask, J, ins, tgs))
    with gpu_context(w, ins, tgs, mask) as ctx:
        ctx.set_controls(u)
        ctx.set_noise(J)
        _, g = ctx.fidelity_grad()
        O = ctx.overlaps()
    return np.ravel(O), g, np.ravel(Oo), go


def _product(vs):
    return synth.MPS([np.asarray(v, dtype=np.complex128).reshape(1, 2, 1) for v in vs])


@pytest.mark.parametrize("sigma", [0.1, 0.03, 0.01, 0.001])
def test_weak_controls_towards_the_opposite_state(sigma):
    """|0..0> to |1..1> on 8 qubits without crosstalk: every site contributes an
    amplitude of the rotation angle, |O| from 1e-14 down to 1e-30.  A site's
    amplitude (2e-4 at the weakest) carries the rounding of about 100 gates, 1e-16
    each: 5e-11 of it, eight sites 4e-10, below the bar of 1e-8."""
    w = synth.WORKLOADS["x8"].replace(M=1, P=1)
    u = np.random.default_rng(5).normal(0.0, sigma, size=(w.K, w.C, w.N))
    O, g, Oo, go = _both(w, u, np.zeros((1, w.N - 1)), [_product([[1, 0]] * w.N)], [_product([[0, 1]] * w.N)])
    assert abs(O[0] - Oo[0]) <= TOL_G_REL * abs(Oo[0])
    assert grad_close(g, go)


@pytest.mark.parametrize("flips", [(2, 3), (1, 2, 4, 5)])
@pytest.mark.parametrize("eps", [1e-3, 1e-5])
def test_target_reached_only_through_weak_couplings(eps, flips):
    """The target is the uncoupled evolution with neighbouring sites turned to the
    orthogonal state, so only the Schmidt components that couplings of eps create
    reach it: |O| is about eps for one pair, eps^2 for two.  The couplings enter the
    gates as 0.3 eps beside roundings of 4e-16, twelve gates deep: 5e-10 of a
    component at eps = 1e-5, below the bar of 1e-8."""
    w = synth.WORKLOADS["x8"].replace(N=7, K=3, dt=0.3, chi=8, M=1, P=1)
    rng = np.random.default_rng(7)
    u = np.zeros((w.K, w.C, w.N))
    u[:, 0] = 0.3
    u[:, 1] = 0.2 * rng.normal(size=(w.K, w.N))
    z = rng.normal(size=(w.N, 2)) + 1j * rng.normal(size=(w.N, 2))
    z /= np.linalg.norm(z, axis=1, keepdims=True)
    J = eps * (1.0 + rng.uniform(0.0, 1.0, size=(1, w.N - 1)))
    X, Y = np.array([[0, 1], [1, 0]]), np.array([[0, -1j], [1j, 0]])
    tgt = []
    for i in range(w.N):
        v = z[i]
        for k in range(w.K):
            x, y = w.dt * u[k, :, i]
            a = np.hypot(x, y)
            v = np.cos(a) * v - 1j * np.sin(a) / a * ((x * X + y * Y) @ v)
        tgt.append([-np.conj(v[1]), np.conj(v[0])] if i in flips else v)
    O, g, Oo, go = _both(w, u, J, [_product(z)], [_product(tgt)])
    assert abs(Oo[0]) < 2 * (2 * eps) ** (len(flips) // 2)
    assert abs(O[0] - Oo[0]) <= TOL_G_REL * abs(Oo[0])
    assert grad_close(g, go)


@pytest.mark.parametrize("N,chi,seed,same", [(16, 20, 2, True), (24, 24, 1, True), (24, 24, 1, False)])
def test_dense_operators(N, chi, seed, same):
    """Random dense operators as input and target, alike or unrelated: every bond is
    full and the environments' sums have chi terms of one size."""
    w = synth.WORKLOADS["cnotgate50"].replace(N=N, K=1, C=2, chi=chi, M=1, P=1, dt=0.1)
    rng = np.random.default_rng(seed)
    D = [min(chi, 4 ** min(i, 6), 4 ** min(N - i, 6)) for i in range(N + 1)]
    op = [synth.MPS([(rng.normal(size=(D[i], 4, D[i + 1])) + 1j * rng.normal(size=(D[i], 4, D[i + 1])))
                     / np.sqrt(8.0 * D[i + 1]) for i in range(N)]) for _ in range(2)]
    u = rng.normal(0.0, 0.5, size=(w.K, w.C, N))
    J = rng.uniform(-0.1, 0.1, size=(1, N - 1))
    _, g, _, go = _both(w, u, J, [op[0]], [op[0] if same else op[1]])
    assert grad_close(g, go)
