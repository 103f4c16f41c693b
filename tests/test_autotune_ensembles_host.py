"""The cached launch shape and the ensemble's size, on the CPU: a shape tuned on an
ensemble that fills two CTAs per SM is not taken for one that does not fill one."""
import json

import pytest

from paper_2603_03639_gb300 import autotune


@pytest.fixture()
def path(tmp_path):
    p = tmp_path / "tuned.json"
    p.write_text(json.dumps({
        "N50-C3-K128-T2048-chi64-grad": {"warps": 4, "ctas_per_sm": 2, "pairs": False},
        "N30-C3-K128-T256-chi64-grad": {"warps": 4, "ctas_per_sm": 2, "pairs": False, "trajectories": 200},
        "N20-C3-K128-T256-chi64-grad": {"warps": 6, "ctas_per_sm": 1, "pairs": False, "trajectories": 140},
    }))
    return str(p)


@pytest.mark.parametrize("M,shape", [(1, (0, 0)), (19, (0, 0)), (20, (4, 2)), (256, (4, 2)), (4096, (4, 2))])
def test_nearest_bucket_on_the_same_side_of_the_sms(path, M, shape):
    args = (50, 100, 64, M, 8, 3)
    assert autotune.lookup(*args, path=path) == shape
    assert autotune.lookup_pairs(*args, path=path) is (shape == (0, 0))


@pytest.mark.parametrize("N,M,shape", [(30, 150, (0, 0)), (30, 160, (4, 2)), (20, 150, (6, 1)), (20, 160, (0, 0)),
                                       (20, 16, (6, 1))])
def test_a_bucket_across_the_sms_goes_by_the_ensemble_it_was_tuned_on(path, N, M, shape):
    assert autotune.lookup(N, 100, 64, M, 1, 3, path=path) == shape


def test_every_warp_count_is_timed_on_short_chains(monkeypatch):
    """All warps share a CTA's environments and large bonds, so the default of eight is
    a candidate on four bonds a layer too."""
    from paper_2603_03639_gb300 import tnrc
    made = []

    class Context:
        def __init__(self, *a, warps, ctas_per_sm, **kw):
            made.append((warps, ctas_per_sm))

        def __enter__(self):
            return self

        def __exit__(self, *a):
            return False

        def stats(self):
            return {"traj_ms": 1.0, "traj_launches": 1}

        def __getattr__(self, name):
            return lambda *a: None
    monkeypatch.setattr(tnrc, "Context", Context)
    best, times = autotune.tune(8, 4, 0.1, 16, 4, 2, [None], [None], None, (1, 0, 0.1), candidates=autotune.QUICK)
    assert [m for m in made[:len(autotune.QUICK)]] == autotune.QUICK
    assert best[0] * best[1] <= 16 and len(times) == len(autotune.QUICK) + 2
