"""The AMG solvers' waits for the parts of their operators, given up on request (wait_timeout 0): every
kernel form leaves with AVIP_ETIMEOUT in the run's and the solve's status, with its copies in flight
waited for, and the same handle then matches the oracle.  One thread-block cluster with the inverse, the
V-cycle from shared memory or streamed; the whole GPU; a single block; mixed precision; a batch."""
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


def _problem(nx, ny, axisym=False):
    kw = dict(field_dependent=True, source=W.SRC_TOWNSEND)
    if axisym:
        return W.axisym_problem(nx, ny, 1.25e-2, 1.25e-2, 18750.0, seed=nx, n_peak=5e18, n_back=1e13, sigma=4e-4,
                                x0=1e-2, **kw)
    return W.plates_problem(nx, ny, 1e-2, 1e-2, 1e4, seed=nx + ny, **kw)


def _matches(m, p, steps, tol):
    n, phi, _ = O.Oracle(p).run(steps)
    for s in range(2):
        assert normwise(m.density(s), n[s]) <= tol
    assert normwise(m.phi(), phi) <= tol


@pytest.mark.parametrize("nx,ny,kind,expect,mixed,axisym", [
    (17, 17, 0, 11, False, False), (40, 45, 11, 11, False, False), (121, 117, 11, 11, False, False),
    (57, 64, 0, 8, False, False), (11, 9, 8, 8, False, False), (121, 117, 8, 8, False, False),
    (9, 11, 9, 9, False, True), (61, 73, 9, 9, False, True),
    (35, 31, 11, 11, True, False), (13, 19, 10, 10, True, False), (121, 117, 10, 10, True, False)])
def test_wait_given_up_then_handle_recovers(avip, nx, ny, kind, expect, mixed, axisym):
    p = _problem(nx, ny, axisym)
    kw = dict(precision=avip.PREC_MIXED, rtol=1e-10) if mixed else dict(rtol=1e-13)
    m = avip.Mesh(p, pcg_kind=kind, wait_timeout=0.0, **kw)
    assert m.info["pcg_kind"] == expect
    s0 = m.state()
    for _ in range(2):
        st = m.run(1, allow=(avip.AVIP_ETIMEOUT,))
        assert st["status"] == avip.AVIP_ETIMEOUT
        rc, _, _ = avip.poisson_solve(m.h)
        assert rc == avip.AVIP_ETIMEOUT
    m.set_wait_timeout(2.0)
    m.set_state(s0)
    assert m.run(2)["steps"] == 2
    _matches(m, p, 2, 1e-6 if mixed else 1e-10)
    m.close()


@pytest.mark.parametrize("mixed", [False, True])
def test_wait_given_up_in_a_batch(avip, mixed):
    """One instance of three gives up; the others end as the oracle does."""
    ps = [_problem(23, 19), _problem(41, 37), _problem(61, 53)]
    kw = dict(precision=avip.PREC_MIXED, rtol=1e-10, pcg_kind=11) if mixed else dict(rtol=1e-13, pcg_kind=11)
    meshes = [avip.Mesh(p, wait_timeout=0.0 if k == 1 else 2.0, **kw) for k, p in enumerate(ps)]
    b = avip.Batch(meshes, cluster_size=16)
    st = b.run(2, allow=(avip.AVIP_ETIMEOUT,))
    assert [s["status"] for s in st] == [avip.AVIP_OK, avip.AVIP_ETIMEOUT, avip.AVIP_OK]
    for k in (0, 2):
        _matches(meshes[k], ps[k], 2, 1e-6 if mixed else 1e-10)
    b.close()
    for m in meshes:
        m.close()
