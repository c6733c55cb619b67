"""Small planar FP64 meshes are solved with the inverse of the matrix as the preconditioner
(dense_inverse.cu); sizes at the edges of its 64-row tiles, of its switch from one cluster to the
whole GPU, of a row per warp and of its range, against the oracle's direct solve.  And the FP32
screening of the cell time step against the oracle on densities that span twenty decades."""
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


@pytest.mark.parametrize("nx,ny,kind", [
    (3, 3, 11), (8, 8, 11), (13, 5, 11), (16, 8, 11), (43, 3, 11), (30, 40, 11), (27, 45, 8), (57, 64, 8), (50, 73, 8),
    (64, 72, 8), (11, 419, 11)])
def test_direct_preconditioner_sizes(avip, nx, ny, kind):
    p = W.plates_problem(nx, ny, 1e-2, 1e-2, 5e3, seed=nx + ny, field_dependent=True, source=W.SRC_TOWNSEND)
    o = O.Oracle(p)
    m = avip.Mesh(p, rtol=1e-12)
    assert m.info["pcg_kind"] == kind
    it, rr = m.poisson_solve()
    phi = o.poisson(o.initial_state())
    assert rr <= 1e-12
    assert normwise(m.phi(), phi) <= 1e-10
    if nx * ny <= 4608:   # an FP32 inverse leaves two or three iterations (4 bounds a poor one)
        assert it <= 4, it
    m2 = avip.Mesh(p, rtol=1e-12)
    m2.run(3)
    n, _, _ = o.run(3)
    for s in range(2):
        assert normwise(m2.density(s), n[s]) <= 1e-10


@pytest.mark.parametrize("nx,ny,lx,kind", [(4, 100, 1e-4, 5), (25, 50, 3e-4, 11), (30, 45, 1e-3, 11)])
def test_ill_conditioned_matrices_keep_their_solver(avip, nx, ny, lx, kind):
    """Cells of aspect 50 and more between electrodes at the long ends: the FP32 inverse is
    rejected (spectral bound above 1/2) and the solve converges as without it.  Error of the
    scaled potential: at most the residual over the smallest eigenvalue (twice that, for the
    rounding of the oracle's solution at these conditions)."""
    rtol = 1e-10
    p = W.plates_problem(nx, ny, lx, 1.0, 5e3, seed=nx + ny)
    o = O.Oracle(p)
    free = p.node_bc != 1
    K = o.K.toarray()[free][:, free]
    d = np.sqrt(np.diag(K))
    phi = o.poisson(o.initial_state())
    b = (K @ phi[free]) / d
    A = K / np.outer(d, d)
    M = np.linalg.inv(A.astype(np.float32)).astype(np.float64)
    assert np.abs(A @ ((M + M.T) / 2) - np.eye(len(A))).sum(1).max() > 0.5
    m = avip.Mesh(p, rtol=rtol)
    assert m.info["pcg_kind"] == kind
    it, rr = m.poisson_solve()
    assert rr <= rtol
    err = np.linalg.norm(d * (m.phi() - phi)[free])
    assert err <= 2 * rtol * np.linalg.norm(b) / np.linalg.eigvalsh(A)[0]


@pytest.mark.parametrize("quads,ns,seed", [(0.0, 2, 1), (0.0, 3, 2), (0.5, 2, 3), (1.0, 3, 4)])
def test_time_step_screening(avip, quads, ns, seed):
    """The step equals the oracle's minimum with densities from 1e0 to 1e20, a few of them
    negative, and velocities of opposite signs around the seed."""
    rng = np.random.default_rng(seed)
    kw = dict(field_dependent=True, source=W.SRC_TOWNSEND_ATTACH if ns == 3 else W.SRC_TOWNSEND, n_species=ns)
    if quads > 0:
        p = W.hybrid_plates_problem(37, 41, 1e-2, 1e-2, 1e4, seed, quad_fraction=quads, **kw)
    else:
        p = W.plates_problem(37, 41, 1e-2, 1e-2, 1e4, seed, **kw)
    sp = []
    for s in p.species:
        n0 = 10.0 ** rng.uniform(0.0, 18.0, p.n_nodes) * np.where(rng.uniform(size=p.n_nodes) < 0.05, -1.0, 1.0)
        sp.append(dataclasses.replace(s, n0=n0))
    p = dataclasses.replace(p, species=sp)
    o = O.Oracle(p)
    _, info = o.step(o.initial_state())
    m = avip.Mesh(p, rtol=1e-13)
    dt = m.step()
    assert abs(dt - info["dt"]) <= 1e-10 * info["dt"]  # (max |E| carries the solve tolerance)
