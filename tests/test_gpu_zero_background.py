"""Densities on a zero background: an explicit front that runs into it decays through the subnormal
numbers (an edge's difference below 2^-1024 has no finite reciprocal), and the step stays that of the
oracle."""
import numpy as np
import pytest

import avip_oracle as O
from helpers import normwise
from paper_2201_01291_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def avip():
    from paper_2201_01291_gb300 import avip as m
    m.load()
    return m


def _pulse(nx, **opts):
    return W.plates_problem(nx, nx, 1e-2, 1e-2, 5e3, seed=5, n_back=0.0, sigma=2e-4, field_dependent=True,
                            source=W.SRC_TOWNSEND, opts=W.Opts(**opts))


def _smallest_difference(o, n):
    d = np.abs(n[o.edges[:, 1]] - n[o.edges[:, 0]])
    return d[d > 0].min()


@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("limiter,beta", [(W.LIM_SWEBY, 1.0), (W.LIM_SWEBY, 1.5), (W.LIM_VANLEER, 1.0)])
def test_limiter_on_subnormal_differences(avip, limiter, beta, batch):
    p = _pulse(129, limiter=limiter, beta=beta)
    o = O.Oracle(p)
    n, phi, _ = o.run(4)
    assert _smallest_difference(o, n[0]) < 2.0 ** -1024  # the case is reached
    m = avip.Mesh(p, rtol=1e-13)
    if batch:
        b = avip.Batch([m], cluster_size=16)
        b.run(4)
        b.close()
    else:
        assert m.run(4)["status"] == avip.AVIP_OK
    for s in range(2):
        assert np.all(np.isfinite(m.density(s)))
        assert normwise(m.density(s), n[s]) <= 1e-10
    assert normwise(m.phi(), phi) <= 1e-10
    m.close()
