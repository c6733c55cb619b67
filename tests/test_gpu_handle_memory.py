"""Device memory a handle holds (mesh_info), and what creating one does when memory runs short."""
import dataclasses

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


@pytest.mark.parametrize("nx,ny,kind", [(95, 95, 0), (65, 65, 11)])
def test_fp64_handles_hold_only_a_tail_they_apply(avip, nx, ny, kind):
    """One cluster of 16 CTAs applies a tail of at most 4.2 MB (256 KB each); some 1,500 bytes a node beside."""
    m = avip.Mesh(_plates(nx, ny), pcg_kind=kind)
    assert m.info["pcg_kind"] == 11
    assert m.info["device_bytes"] <= 1600 * nx * ny + 16 * 256 * 1024
    m.close()


@pytest.mark.parametrize("nx,ny,lx,kind", [(4, 100, 1e-4, 5), (25, 50, 3e-4, 11), (30, 45, 1e-3, 11)])
def test_a_rejected_inverse_is_given_back(avip, nx, ny, lx, kind):
    """Meshes too ill-conditioned for an FP32 inverse: as many bytes as with their solver asked for."""
    p = W.plates_problem(nx, ny, lx, 1.0, 5e3, seed=nx + ny)
    m, f = avip.Mesh(p), avip.Mesh(p, pcg_kind=kind)
    assert m.info["pcg_kind"] == f.info["pcg_kind"] == kind
    assert m.info["device_bytes"] == f.info["device_bytes"]
    m.close()
    f.close()


@pytest.mark.parametrize("nx,ny,largest,kind", [(65, 65, 60e6, 11), (65, 65, 2e6, 11), (20, 23, 5e5, 5)])
def test_no_memory_for_the_inverse(avip, monkeypatch, nx, ny, largest, kind):
    """An allocator that gives no block above `largest` bytes: the handle does without the inverse, which
    only speeds its solves up."""
    inner, free = avip.torch_allocator()
    refused = []

    @avip.ALLOC_FN
    def alloc(nbytes, ctx):
        if nbytes > largest:
            refused.append(nbytes)
            return None
        return inner(nbytes, ctx)

    monkeypatch.setattr(avip, "torch_allocator", lambda: (alloc, free))
    p = _plates(nx, ny)
    m = avip.Mesh(p, rtol=1e-13, use_torch_allocator=True)
    assert refused and m.info["pcg_kind"] == kind
    m.run(3)
    n, phi, _ = O.Oracle(p).run(3)
    for s in range(2):
        assert normwise(m.density(s), n[s]) <= 1e-10
    assert normwise(m.phi(), phi) <= 1e-10
    m.close()


@pytest.mark.parametrize("nx,ny", [(31, 37), (65, 65)])
def test_handles_with_the_inverse_hold_no_hierarchy(avip, nx, ny):
    """Less than the inverse (64-row tiles) beside a handle of the V-cycle, which has its levels."""
    p = _plates(nx, ny)
    m, f = avip.Mesh(p), avip.Mesh(p, pcg_kind=11)
    rows = (nx * ny + 63) // 64 * 64
    assert len(f.info["levels"]) > 1
    assert m.info["levels"] == [(nx * ny, m.info["nnz"], 0, 0, 0, 0)]
    assert m.info["device_bytes"] < f.info["device_bytes"] + 4 * rows * rows
    m.close()
    f.close()


@pytest.mark.parametrize("nx,ny,cluster", [
    (16, 32, 2), (27, 19, 2), (31, 37, 2), (31, 37, 16), (32, 48, 16), (29, 53, 16), (65, 65, 0), (65, 65, 2)])
def test_inverse_in_a_batch(avip, nx, ny, cluster):
    """512 and 513 rows: the last that two CTAs apply and the first that they do not; 1,536 and 1,537: likewise
    for 16.  Above, no batch can, and the inverse is given back.  The handle then still steps on its own."""
    p, q = _plates(nx, ny), _plates(17, 17)
    m, other, f = avip.Mesh(p, rtol=1e-13), avip.Mesh(q, rtol=1e-13), avip.Mesh(p, pcg_kind=11)
    b = avip.Batch([m, other], cluster_size=cluster)
    if nx * ny > 1536:
        # (the solver's partials and flags are those of the whole GPU)
        assert avip.mesh_info(m.h)["device_bytes"] <= f.info["device_bytes"] + (1 << 15)
    b.run(2)
    b.close()
    for mesh, prob in ((m, p), (other, q)):
        mesh.run(2)
        n, phi, _ = O.Oracle(prob).run(4)
        for s in range(2):
            assert normwise(mesh.density(s), n[s]) <= 1e-10
        assert normwise(mesh.phi(), phi) <= 1e-10
    for h in (m, other, f):
        h.close()


@pytest.mark.parametrize("n", [7, 21, 37, 67, 95, 201])
@pytest.mark.parametrize("mesh", ["triangles", "quads", "mixed cells", "axisym", "photo", "axisym photo"])
def test_serving_reserves_what_a_handle_holds(avip, n, mesh):
    """A request's estimate covers the handle it is served with, and is not twice as much beside the dense
    operators and a megabyte."""
    from paper_2201_01291_gb300 import serve
    kw = dict(field_dependent=True, source=W.SRC_TOWNSEND)
    axisym = mesh.startswith("axisym")
    if axisym:
        p = W.axisym_problem(n, n, 1.25e-2, 1.25e-2, 18750.0, seed=n, n_peak=5e18, n_back=1e13, sigma=4e-4,
                             x0=1e-2, **kw)
    elif mesh in ("quads", "mixed cells"):
        p = W.hybrid_plates_problem(n, n, 1e-2, 1e-2, 1e4, n, quad_fraction=1.0 if mesh == "quads" else 0.5, **kw)
    else:
        p = W.plates_problem(n, n, 1e-2, 1e-2, 5e3, seed=n, **kw)
    if mesh.endswith("photo"):
        p = dataclasses.replace(p, photo=W.photo_air())
    for prec in (avip.PREC_FP64,) if axisym or p.photo is not None else (avip.PREC_FP64, avip.PREC_MIXED):
        m = avip.Mesh(p, pcg_kind=serve.solver_kind(p, prec), cluster_size=serve.cluster_ctas(p), precision=prec)
        held, reserved = avip.mesh_info(m.h)["device_bytes"], serve.estimate_bytes(p, prec)
        m.close()
        dense = 4 * 4 * min(p.n_nodes, serve.DENSE_ROWS) ** 2
        assert held <= reserved <= 2 * held + dense + (1 << 20), (prec, held, reserved)
