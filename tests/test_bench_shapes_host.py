"""The launch shape that bench.py measures the plain paths against, on the CPU with a
stand-in context."""
import argparse
import importlib.util
import json
import os

import numpy as np
import pytest

import synth

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture()
def bench():
    spec = importlib.util.spec_from_file_location("bench", os.path.join(HERE, "..", "bench.py"))
    m = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(m)
    return m


def test_plain_sample_runs_in_its_own_shape(bench, monkeypatch, capsys):
    """16 trajectories do not run in the shape cached for 2048."""
    import torch

    import paper_2603_03639_gb300 as pkg
    shapes = []

    class Context:
        def __init__(self, *a, warps, ctas_per_sm, **kw):
            shapes.append((warps, ctas_per_sm))

        def fidelity_grad(self):
            return 0.5, np.zeros(1)

        fidelity_grad_plain = fidelity_grad

        def __getattr__(self, name):
            return lambda *a: None
    monkeypatch.setattr(pkg, "Context", Context)
    monkeypatch.setattr(torch.cuda, "synchronize", lambda *a: None)
    bench.plain_arm(argparse.Namespace(plain_samples=2, steps=1), synth.WORKLOADS["cnot50"])
    line = json.loads(capsys.readouterr().out.splitlines()[-1])
    assert shapes == [(0, 0)] * 3
    assert line["launch_shape"] == {"warps_per_cta": "default", "ctas_per_sm": "default"}
