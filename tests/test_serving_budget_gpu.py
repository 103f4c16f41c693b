"""A server whose budget does not hold a request's default context serves it with one
CTA per SM."""
import numpy as np
import pytest

import synth
from oracle import noise
from tests._util import gpu_context

pytestmark = pytest.mark.gpu


def test_request_beyond_its_share_runs_with_one_cta_per_sm():
    from paper_2603_03639_gb300.serving import Request, Server
    w = synth.WORKLOADS["x8"].replace(N=16, K=12, chi=16, M=400, P=1)
    ins, tgs = w.states()
    req = Request(key="a", N=w.N, K=w.K, dt=w.dt, chi=w.chi, M=w.M, C=w.C, inputs=ins, targets=tgs, controls=w.controls(),
                  noise_seed=5, noise_dist=0, noise_scale=0.05, mask=w.mask())
    one, default = req.footprint(warps=8, ctas_per_sm=1), req.footprint()
    assert one < default
    srv = Server(mem_budget=(one + default) // 2, max_inflight=4)
    srv.submit(req)
    srv.drain()
    srv.close()
    assert req.error is None
    with gpu_context(w, ins, tgs, w.mask(), warps=8, ctas_per_sm=1) as ctx:
        ctx.set_controls(w.controls())
        ctx.set_noise(noise.sample_J(5, w.M, w.N, 0, 0.05))
        F, g = ctx.fidelity_grad()
    assert req.F == F and np.array_equal(req.grad, g)
