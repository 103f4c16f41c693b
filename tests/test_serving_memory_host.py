"""The launch shape that the server asks for, by its memory budget, on the CPU."""
import numpy as np
import pytest

from paper_2603_03639_gb300 import build
from paper_2603_03639_gb300.serving import Request


def _request(M, P, N=50, K=64, chi=32):
    return Request(key="x", N=N, K=K, dt=0.05, chi=chi, M=M, C=2, inputs=[None] * P, targets=[None] * P,
                   controls=np.zeros((K, 2, N)), noise_seed=1, noise_dist=0, noise_scale=0.1)


@pytest.fixture(scope="module", autouse=True)
def library():
    build.build()


def test_half_the_regions_where_the_default_exceeds_its_share():
    r = _request(128, 8)
    default, one = r.footprint(), r.footprint(warps=8, ctas_per_sm=1)
    assert one < 0.6 * default
    assert r.shape(default) == {}
    assert r.footprint(**r.shape(default - 1)) == one


def test_the_default_where_one_cta_per_sm_takes_no_less():
    """160 trajectories of a short chain at chi = 64: 152 regions with eight warps'
    scratch outweigh 160 with four's."""
    r = _request(160, 1, N=10, K=4, chi=64)
    assert r.footprint(warps=8, ctas_per_sm=1) > r.footprint()
    assert r.shape(0) == {}


def test_requests_of_few_trajectories_take_one_shape():
    r = _request(8, 2)
    assert r.footprint() == r.footprint(**r.shape(0))
