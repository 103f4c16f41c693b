"""The integer SVD and the ways a layer's bonds are shared out, against the
oracle at the sizes where they change: bonds of one (theta 2 x 2 at the chain's
ends), two bonds per warp from 33 sites on, updates shared by the CTA's warps
(from theta sides of 16, in shared memory and, wider, in global scratch), the
operator form, and components of very different weight."""
import numpy as np
import pytest

import synth
from oracle import robust
from tests._util import TOL_F, TOL_O, case, gpu_context, grad_close, oracle_problem

pytestmark = pytest.mark.gpu


def _check(w, u=None, warps=0, ctas=0):
    u, mask, J, ins, tgs = case(w, u)
    Fo, go, Oo = robust.ensemble(oracle_problem(w, u, mask, J, ins, tgs))
    with gpu_context(w, ins, tgs, mask, warps=warps, ctas_per_sm=ctas) as ctx:
        ctx.set_controls(u)
        ctx.set_noise(J)
        F, g = ctx.fidelity_grad()
        O = ctx.overlaps()
        st = ctx.stats()
    assert abs(F - Fo) <= TOL_F
    assert np.max(np.abs(O - Oo)) <= TOL_O
    assert grad_close(g, go)
    return st


@pytest.mark.parametrize("N", [2, 3, 32, 33, 34])
def test_bonds_per_warp(N):
    _check(synth.WORKLOADS["x8"].replace(N=N, K=3, dt=0.2, chi=8, M=2, P=1, u_sigma=1.0, target="input"))


@pytest.mark.parametrize("N,chi,K", [(8, 16, 4), (9, 15, 4), (11, 31, 4), (13, 64, 5)])
@pytest.mark.parametrize("shape", [(0, 0), (2, 1), (4, 4)])
def test_updates_shared_by_the_cta(N, chi, K, shape):
    """theta sides of 16 to 128, odd caps; the last case leaves shared memory."""
    w = synth.WORKLOADS["ghz30"].replace(N=N, K=K, chi=chi, M=1, P=1, u_sigma=1.5, dt=0.4)
    st = _check(w, warps=shape[0], ctas=shape[1])
    assert st["max_bond"] > chi // 2


@pytest.mark.parametrize("N,chi", [(3, 16), (5, 13), (6, 32)])
def test_operator_form_sizes(N, chi):
    w = synth.WORKLOADS["cnotgate50"].replace(N=N, K=3, chi=chi, M=2, P=1, dt=0.3, u_sigma=1.0, target="x", g_bonds="all")
    _check(w, u=synth.pi_pulse_controls(w.K, w.C, w.N, w.dt, seed=5, jitter=0.3))


@pytest.mark.parametrize("eps", [1e-3, 1e-6, 1e-9])
def test_small_components_keep_their_digits(eps):
    """Weak couplings give Schmidt values eps, eps^2, ..: the gradient of a target
    that only they reach is compared relative to itself."""
    w = synth.WORKLOADS["x8"].replace(N=6, K=3, dt=0.3, chi=8, M=2, P=1, noise_scale=eps, target="input")
    u = np.zeros((w.K, w.C, w.N))
    u[:, 0, :] = 0.3
    _check(w, u=u)
