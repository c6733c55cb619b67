"""Densities on a zero background: an explicit front that runs into it decays through the subnormal
numbers (an edge's difference below 2^-1024 has no finite reciprocal), and the step stays that of the
oracle."""
import dataclasses

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


@pytest.mark.parametrize("batch", [False, True])
def test_bernoulli_function_at_subnormal_arguments(avip, batch):
    """Scharfetter-Gummel fluxes in a field so weak that h V.e / D is subnormal: B = 1, plain
    diffusion.  Tolerance: one explicit step moves a density by less than itself through at most
    ten edges of some ten roundings each, 1e-14."""
    p = W.plates_problem(23, 19, 1e-2, 1e-2, 1e-309, seed=3, opts=W.Opts(scheme=W.FLUX_SG))
    o = O.Oracle(p)
    n0 = o.initial_state()
    _, E, _, _, vel, _ = o.fields(n0)
    d = p.xy[o.edges[:, 1]] - p.xy[o.edges[:, 0]]
    a = np.abs(0.5 * np.einsum("ij,ij->i", vel[0][o.edges[:, 0]] + vel[0][o.edges[:, 1]], d) / p.species[0].D)
    assert np.any((a > 0) & (a < 2.0 ** -1024))
    n, _ = o.step(n0, dt_fixed=1e-8)
    assert np.abs(n[0] - n0[0]).max() > 1e-3 * np.abs(n[0]).max()
    m = avip.Mesh(p, rtol=1e-13, dt_fixed=1e-8)
    if batch:
        b = avip.Batch([m], cluster_size=8)
        b.run(1)
        b.close()
    else:
        assert m.step() == 1e-8
    for s in range(2):
        assert normwise(m.density(s), n[s]) <= 1e-14
    m.close()


@pytest.mark.parametrize("batch", [False, True])
def test_diffusion_without_a_finite_reciprocal(avip, batch):
    """D = 1e-310 (1 / D overflows) in Scharfetter-Gummel fluxes without a field: nothing moves.  Tolerance:
    the update adds nothing to a density, one rounding."""
    p = W.plates_problem(23, 19, 1e-2, 1e-2, 0.0, seed=3, opts=W.Opts(scheme=W.FLUX_SG))
    p = dataclasses.replace(p, species=[dataclasses.replace(s, D=1e-310) for s in p.species])
    o = O.Oracle(p)
    n, _ = o.step(o.initial_state(), dt_fixed=1e-8)
    m = avip.Mesh(p, rtol=1e-13, dt_fixed=1e-8)
    if batch:
        b = avip.Batch([m], cluster_size=8)
        b.run(1)
        b.close()
    else:
        assert m.step() == 1e-8
    for s in range(2):
        assert normwise(m.density(s), n[s]) <= 2.3e-16
    m.close()
