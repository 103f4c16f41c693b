"""Overlaps of two qubits after a few slices against the same product of matrix
exponentials in extended precision."""
import numpy as np
import pytest

import synth
from tests._util import gpu_context

pytestmark = pytest.mark.gpu

LD, CL = np.longdouble, np.clongdouble


def _expm(a):
    """exp(a) by its Taylor series on a / 2^6, squared six times as exp - 1."""
    b, e, t = a / LD(64), np.zeros_like(a), np.eye(len(a), dtype=CL)
    for k in range(1, 25):
        t = t @ b / LD(k)
        e = e + t
    for _ in range(6):
        e = 2 * e + e @ e
    return e + np.eye(len(a), dtype=CL)


def _overlap(u, J, dt, start, target):
    x = np.array([[0, 1], [1, 0]], dtype=CL)
    y = np.array([[0, -1j], [1j, 0]], dtype=CL)
    one, zz = np.eye(2, dtype=CL), np.diag(np.array([1, -1, -1, 1], dtype=CL))
    psi = np.kron(*[s.astype(CL) / np.sqrt((np.abs(s.astype(CL)) ** 2).sum()) for s in start])
    for k in range(len(u)):
        site = [LD(u[k, 0, i]) * x + LD(u[k, 1, i]) * y for i in range(2)]
        psi = _expm(-1j * LD(dt) * (np.kron(site[0], one) + np.kron(one, site[1]) + LD(J) * zz)) @ psi
    t = np.kron(*[s.astype(CL) / np.sqrt((np.abs(s.astype(CL)) ** 2).sum()) for s in target])
    return np.vdot(t, psi)


def test_two_qubits_in_extended_precision():
    """12 slices of random controls, two half-step layers at each end and merged ones
    between, 13 in all.  A layer rounds a gate by 1e-16 of its angle, theta's products by
    1e-16 of themselves, theta to steps of 2^-55 of its rows and the new sites to 2^-56:
    about 1.4e-16 of the state as root mean square, 5e-16 over 13 layers; the bar is half as
    much again.  (Gates right to 3e-16 of one, as eigenvectors of several rotations give
    them, pass it alone.)"""
    if np.finfo(LD).eps > 1e-18:
        pytest.skip("no extended precision")
    w = synth.WORKLOADS["x8"].replace(N=2, K=12, dt=0.05, chi=2, M=1, P=1)
    rng = np.random.default_rng(9)
    off = []
    for _ in range(96):
        u = rng.normal(0.0, 0.5, size=(w.K, 2, 2))
        J = rng.uniform(-0.05, 0.05)
        a, b = (rng.normal(size=(2, 2)) + 1j * rng.normal(size=(2, 2)) for _ in range(2))
        mps = [synth.MPS([s.reshape(1, 2, 1) for s in v]) for v in (a, b)]
        with gpu_context(w, [mps[0]], [mps[1]], np.ones((2, 2), dtype=np.uint8)) as ctx:
            ctx.set_controls(u)
            ctx.set_noise(np.array([[J]]))
            ctx.fidelity()
            off.append(float(abs(np.ravel(ctx.overlaps())[0] - _overlap(u, J, w.dt, a, b))))
    rms = float(np.sqrt(np.mean(np.square(off))))
    assert rms <= 7.5e-16, rms
