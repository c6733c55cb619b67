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
