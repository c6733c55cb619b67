"""Device memory a handle holds (mesh_info), and what creating one does when memory runs short."""
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


def _plates(nx, ny):
    return W.plates_problem(nx, ny, 1e-2, 1e-2, 5e3, seed=nx + ny, field_dependent=True, source=W.SRC_TOWNSEND)


@pytest.mark.parametrize("nx,ny", [(65, 65), (95, 95)])
def test_mixed_handles_hold_no_dense_tail(avip, nx, ny):
    """The mixed-precision solves take the coarsest inverse only: some 1,650 bytes a node of per-node
    arrays, mesh slots and levels (the V-cycle's tail as one matrix would add up to 9.4 MB)."""
    m = avip.Mesh(_plates(nx, ny), precision=avip.PREC_MIXED)
    assert m.info["device_bytes"] <= 1800 * nx * ny
    m.close()
