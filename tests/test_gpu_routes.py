"""Routes through the stage kernels that the other files reach in FP64 or on three axes only:
slabs of grids with one or two active axes (halo planes read by the thin kernels), the FP32
sweeps in every tile order, non-physical cells through each FP32 kernel, grids without an
active axis."""
import numpy as np
import pytest

import oracle
from paper_1607_01105_gb300 import inputs, slab

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU, skipped there
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1607_01105_gb300 import ppml  # noqa: E402

F32, F64 = ppml.PPML_F32, ppml.PPML_F64
O, P, R = ppml.OUTFLOW, ppml.PERIODIC, ppml.REFLECT


@pytest.mark.parametrize("dtype", [F64, F32])
@pytest.mark.parametrize("n,bc,world", [((40, 1, 48), (O, O, P, P, P, P), 2), ((1, 24, 45), (P, P, R, O, O, R), 3),
                                        ((37, 1, 64), (R, R, O, O, O, O), 2), ((1, 1, 128), (O,) * 6, 2),
                                        ((1, 1, 96), (P,) * 6, 3)])
def test_slabs_of_thin_grids_equal_the_single_grid(n, bc, world, dtype):
    """The state bit for bit (slabs start on tile boundaries), the maxima exactly, the sums to
    their order."""
    pb = (inputs.random_rough if dtype == F64 else inputs.random_smooth)(n=n, bc=bc)
    u = ppml.to_device(pb.u, dtype)
    v = [torch.empty_like(x) for x in u]
    grid = ppml.Grid(n, pb.h, pb.gamma, pb.cfl, bc, dtype, u0=u)
    for _ in range(3):
        grid.step(u, v, 0.0)
        u, v = v, u
    d = grid.diag()
    Ls = [slab.SlabLayout(n, bc, world, r) for r in range(world)]
    td, rho_ref = ppml.torch_dtype(dtype), oracle.mean_density(pb.u)
    st = [slab.Stages(ppml, L, pb.h, pb.gamma, pb.cfl, dtype,
                      [slab.pad_field(L, a, td, "cuda") for a in pb.u], rho_ref) for L in Ls]
    comm = slab.LocalComm(Ls)
    slab.start(st, comm)
    for _ in range(3):
        slab.step(st, comm, 0.0)
    for L, s in zip(Ls, st):
        ds = s.grid.diag()
        assert (ds["dt_next"], ds["t"], ds["vmax"], ds["cmax"]) == (d["dt_next"], d["t"], d["vmax"], d["cmax"])
        for f in range(6):
            got = L.interior(s.cur[f]).reshape(L.nz, -1)
            assert torch.equal(got, u[f].reshape(n[2], -1)[L.z0:L.z0 + L.nz]), (L.rank, f)
            assert ds["sums"][f] == pytest.approx(d["sums"][f], rel=1e-12, abs=1e-12 * abs(d["sums"][0]))


@pytest.mark.parametrize("bc", [(R, O, P, P, O, R), (P,) * 6])
def test_fp32_tile_orders_give_the_same_bits(bc):
    """x-major, z-major and blocked orders (padded at the ragged edges): the same state, maxima
    and sums over three steps."""
    pb = inputs.random_smooth(n=(53, 37, 41), bc=bc)
    out = []
    for order in range(ppml.TILE_ORDERS):
        u = ppml.to_device(pb.u, F32)
        v = [torch.empty_like(x) for x in u]
        grid = ppml.Grid(pb.n, pb.h, pb.gamma, pb.cfl, bc, F32, u0=u)
        grid.set_order(order)
        for _ in range(3):
            grid.step(u, v, 0.0)
            u, v = v, u
        out.append((u, grid.diag()))
    for u, d in out[1:]:
        assert all(torch.equal(x, y) for x, y in zip(u, out[0][0]))
        assert d == out[0][1]


PLANTED = [(0, -1.0), (0, float("nan")), (1, float("nan")), (2, float("inf")), (4, float("-inf")),
           (5, float("nan"))]


@pytest.mark.parametrize("dtype", [F32, F64])
@pytest.mark.parametrize("n", [(40, 37, 41), (50, 45, 1), (150, 1, 1)])
@pytest.mark.parametrize("field,value", PLANTED)
def test_nonphysical_cells_are_flagged_by_every_kernel(n, dtype, field, value):
    """A cell that is not physical makes the step's count and flag, and stays near its place (a
    step reads three cells each way in each of its two stages); the handle has seen physical
    cells only."""
    pb = inputs.random_smooth(n=n, bc=(O,) * 6)
    u = ppml.to_device(pb.u, dtype)
    v = [torch.empty_like(x) for x in u]
    grid = ppml.Grid(n, pb.h, pb.gamma, pb.cfl, (O,) * 6, dtype, u0=u)
    dt = 0.5 * grid.cfl_dt(u)
    grid.step(u, v, dt)
    assert grid.diag()["n_bad"] == 0
    clean = [x.clone() for x in v]
    bad = [x.clone() for x in u]
    at = [m // 2 if m > 1 else 0 for m in n]
    bad[field].view(n[2], n[1], n[0])[at[2], at[1], at[0]] = value
    grid.step(bad, v, dt)
    d = grid.diag(raise_nonphysical=False)
    assert d["n_bad"] > 0 and d["flags"] & ppml.FLAG_NONPHYSICAL
    with pytest.raises(ppml.PPMLError) as e:
        grid.diag()
    assert e.value.code == ppml.PPML_E_NONPHYSICAL
    z, y, x = np.meshgrid(*[np.abs(np.arange(m) - c) for m, c in zip(n[::-1], at[::-1])], indexing="ij")
    far = torch.as_tensor((np.maximum(np.maximum(x, y), z) > 6).ravel(), device="cuda")
    for a, b in zip(v, clean):
        assert torch.equal(a[far], b[far])


@pytest.mark.parametrize("dtype", [F32, F64])
def test_grid_without_an_active_axis(dtype):
    """One cell: nothing moves, and the internal energy becomes rho E - |m|^2 / (2 rho)."""
    u = [torch.full((1,), a, device="cuda", dtype=ppml.torch_dtype(dtype)) for a in (2.0, 0.5, -0.25, 1.0, 3.0, 2.5)]
    v = [torch.empty_like(x) for x in u]
    grid = ppml.Grid((1, 1, 1), (1.0,) * 3, 1.4, 0.4, (O,) * 6, dtype, u0=u)
    grid.step(u, v, 0.1)
    assert [float(x) for x in v[:5]] == [float(x) for x in u[:5]]
    assert float(v[5]) == 3.0 - 1.3125 / 4.0
    assert grid.diag()["n_bad"] == 0
