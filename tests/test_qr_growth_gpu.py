"""States whose Schmidt values spread over decades: rows of theta grow during the
integer QR and are rescaled, by a half-warp, a warp and the whole CTA, against the
oracle."""
import numpy as np
import pytest

import synth
from oracle import robust
from tests._util import TOL_F, TOL_O, gpu_context, grad_close, oracle_problem

pytestmark = pytest.mark.gpu


def _graded(N, D, decades, rng):
    """A random state of bond dimension D whose left Schmidt vectors at every bond
    carry weights from 1 down to 10^-decades, in steps."""
    dims = [min(D, 2 ** min(i, 10), 2 ** min(N - i, 10)) for i in range(N + 1)]
    sites = []
    for i in range(N):
        a = rng.normal(size=(dims[i], 2, dims[i + 1])) + 1j * rng.normal(size=(dims[i], 2, dims[i + 1]))
        q = np.linalg.qr(a.reshape(dims[i], -1).T)[0].T.reshape(a.shape)   # right-canonical
        lam = 10.0 ** -np.floor(np.linspace(0.0, decades + 0.99, dims[i + 1]))
        sites.append(q * lam)
    return synth.MPS(sites)


@pytest.mark.parametrize("N,chi,decades", [(36, 8, 4), (10, 16, 3), (12, 64, 3), (12, 64, 9), (13, 64, 2)])
def test_graded_states(N, chi, decades):
    w = synth.WORKLOADS["x8"].replace(N=N, K=2, dt=0.1, chi=chi, M=2, P=1, sv_cutoff=1e-12)
    rng = np.random.default_rng(N + decades)
    state = _graded(N, chi, decades, rng)
    u = rng.normal(0.0, 0.3, size=(w.K, w.C, N))
    J = rng.uniform(-0.1, 0.1, size=(w.M, N - 1))
    mask = np.ones((w.C, N), dtype=np.uint8)
    Fo, go, Oo = robust.ensemble(oracle_problem(w, u, mask, J, [state], [state]))
    with gpu_context(w, [state], [state], mask) as ctx:
        ctx.set_controls(u)
        ctx.set_noise(J)
        F, g = ctx.fidelity_grad()
        O = ctx.overlaps()
    assert abs(F - Fo) <= TOL_F
    assert np.max(np.abs(np.ravel(O) - np.ravel(Oo))) <= TOL_O
    assert grad_close(g, go)
