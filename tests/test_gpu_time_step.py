"""The FP32 screening of the cell time step against the oracle's minimum, limit by limit."""
import numpy as np
import pytest

import avip_oracle as O
from paper_2201_01291_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def avip():
    from paper_2201_01291_gb300 import avip as m
    m.load()
    return m


@pytest.mark.parametrize("voltage,seed", [
    (1e-14, 4), (1e-18, 4), (1e-20, 4), (8e-22, 4), (7e-22, 38), (4e-22, 8), (3e-22, 19), (3e-22, 22), (2e-22, 7),
    (2e-22, 11), (2e-22, 20), (2e-22, 37), (1e-23, 4), (1e-30, 4)])
def test_vanishing_fields(avip, voltage, seed):
    """No diffusion and next to no charges: the convective limit alone, down to velocities whose squares are
    subnormal or zero in FP32, in a field that grows across the plates so that fast cells and short
    cells compete.  (max |E| carries the solve tolerance.)"""
    p = W.plates_problem(61, 83, 1e-2, 2e-2, voltage, seed=seed)
    p.phi_D[:] *= 1.0 + 0.8 * p.xy[:, 0] / 1e-2
    for s in p.species:
        s.mob_params, s.D = [2e-4], 0.0
        s.n0[:] = 1e-20 * (1.0 + 0.1 * np.sin(np.arange(p.n_nodes)))
    _, info = O.Oracle(p).step([s.n0 for s in p.species])
    m = avip.Mesh(p, rtol=1e-13)
    dt = m.step()
    assert abs(dt - info["dt"]) <= 1e-10 * info["dt"]
    m.close()


def _neutral(kind, nx, ny, seed, quads, ns):
    """Constant mobilities and neutral pairs (no space charge), so that the dielectric limit sets the
    step whatever the solve's tolerance: densities over twenty decades, nearly equal ones (within the
    screening's margin of 1e-6 of each other), or of either sign, cancelling within the cells."""
    rng = np.random.default_rng(seed)
    if quads > 0:
        p = W.hybrid_plates_problem(nx, ny, 1e-2, 1e-2, 1e4, seed, quad_fraction=quads, n_species=ns)
    else:
        p = W.plates_problem(nx, ny, 1e-2, 1e-2, 1e4, seed, n_species=ns)
    size = p.n_nodes
    if kind == "decades":
        n0 = 10.0 ** rng.uniform(0.0, 20.0, size) * np.where(rng.uniform(size=size) < 0.05, -1.0, 1.0)
    elif kind == "ties":
        n0 = 1e19 * (1.0 + 1e-8 * rng.uniform(-1.0, 1.0, size))
    else:
        n0 = 1e19 * rng.choice([-1.0, 1.0], size) * (1.0 + 0.2 * rng.uniform(size=size))
    p.species[0].n0[:] = n0
    p.species[1].n0[:] = n0
    return p


def _dielectric_limit(p):
    groups = [np.asarray(c) for c in (p.tris, p.quads) if c is not None and len(c)]
    return min(p.opts.a_diel * W.EPS0 / W.E_CHARGE /
               sum(abs((s.n0 * s.mob_params[0])[c].mean(axis=1)) for s in p.species).max() for c in groups)


# (200,000 cells: above four blocks per SM a thread takes several cells)
CASES = [(kind, nx, ny, seed, quads, ns) for kind in ("decades", "ties", "signs") for nx, ny, seed, quads, ns in
         ((9, 7, 1, 0.0, 2), (61, 83, 2, 0.0, 3), (61, 83, 3, 0.5, 2), (33, 29, 4, 1.0, 2), (301, 335, 5, 0.0, 2))]


@pytest.mark.parametrize("kind,nx,ny,seed,quads,ns", CASES)
def test_dielectric_limit(avip, kind, nx, ny, seed, quads, ns):
    """Tolerance: some ten roundings of 1.1e-16 each in FP64; in mixed precision the FP32 mobilities
    (6e-8 each)."""
    p = _neutral(kind, nx, ny, seed, quads, ns)
    want = _dielectric_limit(p)
    o = O.Oracle(p)
    assert abs(o.step(o.initial_state())[1]["dt"] - want) <= 1e-13 * want  # this limit decides
    for precision, tol in ((avip.PREC_FP64, 1e-13), (avip.PREC_MIXED, 2e-7)):
        m = avip.Mesh(p, precision=precision, rtol=1e-10)
        dt = m.step()
        assert abs(dt - want) <= tol * want, precision
        m.close()


@pytest.mark.parametrize("mixed", [False, True])
def test_dielectric_limit_in_a_batch(avip, mixed):
    ps = [_neutral(*c) for c in CASES if c[1] <= 61]
    precision, tol = (avip.PREC_MIXED, 2e-7) if mixed else (avip.PREC_FP64, 1e-13)
    meshes = [avip.Mesh(p, precision=precision, rtol=1e-10) for p in ps]
    b = avip.Batch(meshes, cluster_size=16)
    for threads in (256, 128):
        assert avip.batch_set_dd_threads(b.b, threads) == avip.AVIP_OK
        for m, p in zip(meshes, ps):
            m.set_state(np.concatenate([s.n0 for s in p.species] + [np.zeros(4 * p.n_nodes + 2)]))
        for st, p in zip(b.run(1), ps):
            want = _dielectric_limit(p)
            assert abs(st["dt_min"] - want) <= tol * want
    b.close()
    for m in meshes:
        m.close()
