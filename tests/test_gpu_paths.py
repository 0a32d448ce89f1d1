"""The kernels that a call is routed to by its grid (three active axes, two, one), precision
and size, at the sizes where each can go wrong (edges of tiles and segments, remainders, the
smallest), against the FP64 oracle: FP64 bit for bit, FP32 within the single-step bar 1e-5
(relative L1 per field; a momentum against at least 1e-3 of the density's L1, as it may
vanish)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import oracle  # noqa: E402
from paper_1607_01105_gb300 import inputs, ppml  # noqa: E402

pytestmark = pytest.mark.gpu

F32, F64 = ppml.PPML_F32, ppml.PPML_F64
O, P, R, I = ppml.OUTFLOW, ppml.PERIODIC, ppml.REFLECT, ppml.INFLOW
BAR = 1e-5


def _state(rho, mx, my, mz, p, gamma=1.4):
    ei = p / (gamma - 1.0)
    return (rho, mx, my, mz, ei + 0.5 * (mx * mx + my * my + mz * mz) / rho, ei)


INFLOW = {q: _state(1.0 + 0.1 * q, 0.3 - 0.1 * q, 0.2, 0.05 * q - 0.1, 0.9 + 0.05 * q) for q in range(6)}

FORMS = [
    # three axes: whole tiles, ragged ones with walls on both ends of every axis, the smallest
    ((16, 16, 16), (O, O, P, P, O, R), 0), ((17, 15, 33), (R, O, O, R, R, R), 0),
    ((33, 18, 17), (R,) * 6, 0), ((3, 3, 3), (P,) * 6, 0), ((35, 34, 20), (P, P, R, R, O, O), 1),
    ((20, 37, 18), (O,) * 6, 2), ((19, 17, 18), (I, O, O, I, I, O), 0),
    # two axes
    ((17, 33, 1), (R, O, P, P, O, O), 0), ((16, 1, 16), (P, P, O, O, R, R), 0),
    ((1, 5, 40), (O, O, O, R, P, P), 3), ((37, 20, 1), (I, O, O, I, O, O), 0),
    # one axis
    ((31, 1, 1), (P, P) + (O,) * 4, 0), ((33, 1, 1), (R, R) + (O,) * 4, 0), ((3, 1, 1), (O,) * 6, 0),
    ((1, 65, 1), (O, O, R, O, O, O), 1), ((1, 1, 64), (O,) * 4 + (P, P), 2),
    ((70, 1, 1), (I,) + (O,) * 5, 0),
]


def _problem(n, bc, fp32, rough):
    pb = (inputs.random_rough if rough else inputs.random_smooth)(n=n, bc=bc)
    if fp32:
        pb.u = [a.astype(np.float32).astype(np.float64) for a in pb.u]
    return pb


def _run(pb, dtype, flags, phi=None):
    inflow = {q: INFLOW[q] for q in range(6) if pb.bc[q] == I}
    g = oracle.Grid(pb.n, pb.h, pb.gamma, pb.bc, pb.cfl, rho_mean=oracle.mean_density(pb.u),
                    flags=flags, inflow=inflow)
    dt = oracle.cfl_dt(g, pb.u)
    ref, diag = oracle.step(g, pb.u, dt, phi=phi)
    u = ppml.to_device(pb.u, dtype)
    v = [torch.empty_like(x) for x in u]
    grid = ppml.Grid(pb.n, pb.h, pb.gamma, pb.cfl, pb.bc, dtype, u0=u, flags=flags, inflow=inflow)
    if phi is None:
        grid.step(u, v, dt)
    else:
        grid.step_phi(u, v, ppml.to_device([phi], dtype)[0], dt)
    got = [x.double().cpu().numpy().reshape(ref[0].shape) for x in v]
    return got, ref, grid.diag(), diag


def _fp32_errors(got, ref):
    floor = [0.0 if f in (0, 4, 5) else 1e-3 * np.abs(ref[0]).sum() for f in range(6)]
    return [float(np.abs(got[f] - ref[f]).sum() / max(np.abs(ref[f]).sum(), floor[f])) for f in range(6)]


@pytest.mark.parametrize("n,bc,flags", FORMS)
def test_fp32_step_over_forms(n, bc, flags):
    got, ref, d, dg = _run(_problem(n, bc, True, False), F32, flags)
    err = _fp32_errors(got, ref)
    assert max(err) <= BAR, err
    assert d["dt_next"] == pytest.approx(dg["dt_cfl"], rel=BAR)
    for f in range(6):
        assert d["sums"][f] == pytest.approx(dg["sums"][f], rel=1e-6, abs=1e-6 * abs(dg["sums"][0]))


@pytest.mark.parametrize("n,bc,flags", [x for x in FORMS if 1 in x[0]])
def test_fp64_step_over_thin_forms_bit_for_bit(n, bc, flags):
    got, ref, d, dg = _run(_problem(n, bc, False, True), F64, flags)
    assert [int(np.count_nonzero(got[f] != ref[f])) for f in range(6)] == [0] * 6
    assert d["vmax"] == dg["vmax"] and d["cmax"] == dg["cmax"]


@pytest.mark.parametrize("dtype", [F32, F64])
@pytest.mark.parametrize("n,bc", [((18, 17, 33), (P, P, O, R, O, O)), ((16, 16, 16), (R, O, P, P, P, P)),
                                  ((21, 18, 1), (P, P, O, O, O, O)), ((40, 1, 1), (O,) * 6)])
def test_gravity_step_over_forms(dtype, n, bc):
    pb = _problem(n, bc, dtype == F32, False)
    z, y, x = np.meshgrid(*[np.arange(m) / m for m in n[::-1]], indexing="ij")
    phi = np.sin(2 * np.pi * x) + 0.5 * np.cos(2 * np.pi * (y + z))
    phi = phi.astype(np.float32).astype(np.float64)
    got, ref, _, _ = _run(pb, dtype, 0, phi)
    if dtype == F64:
        assert [int(np.count_nonzero(got[f] != ref[f])) for f in range(6)] == [0] * 6
    else:
        err = _fp32_errors(got, ref)
        assert max(err) <= BAR, err


def test_fp32_noalloc_step_in_several_launches():
    """More tiles than the fixed buffer's face velocities hold (228 of 64): the same bits as the
    handle's step."""
    pb = _problem((17, 17, 907), (O, O, P, P, O, O), True, False)
    u = ppml.to_device(pb.u, F32)
    a, b = [torch.empty_like(x) for x in u], [torch.empty_like(x) for x in u]
    grid = ppml.Grid(pb.n, pb.h, pb.gamma, pb.cfl, pb.bc, F32, u0=u)
    dt = 0.8 * grid.cfl_dt(u)
    grid.step(u, a, dt)
    desc = ppml.make_desc(pb.n, pb.h, pb.gamma, pb.cfl, pb.bc, F32)
    out = ppml.step_noalloc(desc, u, b, dt, oracle.mean_density(pb.u))
    for f in range(6):
        assert torch.equal(a[f], b[f]), f
    d = grid.diag()
    assert out[0] == d["dt_next"] and out[3] == d["sums"]


# the largest matrix that the dense transforms hold is 256 x 256
@pytest.mark.parametrize("n", [(3, 3, 4), (15, 16, 17), (64, 65, 33), (129, 32, 31), (256, 5, 6), (257, 5, 6)])
def test_isolated_poisson_fp32_sizes(n):
    """The FP32 isolated solve within its bar (2e-5 of the largest potential) of the oracle."""
    from oracle import poisson
    h = 0.05
    z, y, x = np.meshgrid(*[(np.arange(m) + 0.5 - 0.5 * m) * h for m in n[::-1]], indexing="ij")
    rho = np.exp(-(x * x / 0.3 + (y - 0.02) ** 2 / 0.2 + z * z / 0.1)).astype(np.float32).astype(np.float64)
    ref = poisson.solve_isolated(rho, h, 1.1)
    u = ppml.to_device([rho] * 6, F32)
    grid = ppml.Grid(n, (h, h, h), 1.4, 0.2, (O,) * 6, F32, u0=u)
    phi = torch.empty_like(u[0])
    grid.poisson_isolated(u[0], phi, 1.1)
    got = phi.double().cpu().numpy().reshape(ref.shape)
    assert np.max(np.abs(got - ref)) <= 2e-5 * np.max(np.abs(ref))


@pytest.mark.parametrize("threads,split", [(256, 0), (512, 0), (1024, 0), (512, 64)])
def test_fp32_batch_of_small_and_uneven_instances(threads, split):
    """Instances of a few cells up to a few runs per thread, whole and split, to their own end
    times (the last step clipped): the oracle's step count within one and its fields within
    the batched bar 1e-4."""
    ncells = [4, 5, 7, 8, 31, 32, 33, 63, 64, 65, 255, 256, 257, 513, 1030]
    gamma, cfl = 1.4, 0.4
    off = np.concatenate([[0], np.cumsum(ncells)])
    u = [np.empty(off[-1]) for _ in range(4)]
    for i, n in enumerate(ncells):
        x = (np.arange(n) + 0.5) / n
        rho = np.where(x < 0.5, 1.0, 0.4 + 0.02 * i)
        v = np.where(x < 0.5, 0.1, -0.05 * (i % 3))
        p = np.where(x < 0.5, 1.0, 0.3)
        ei = p / (gamma - 1.0)
        for k, a in enumerate((rho, rho * v, ei + 0.5 * rho * v * v, ei)):
            u[k][off[i]:off[i + 1]] = a
    t_end = [0.05 + 0.003 * i for i in range(len(ncells))]
    b = ppml.Batch(ncells, [1.0 / n for n in ncells], t_end, gamma, cfl, F32)
    b.set_threads(threads)
    b.set_split(split)
    st = [torch.as_tensor(a).to("cuda", torch.float32) for a in u]
    while b.step(st, 100, sync=True) < len(ncells):
        pass
    t, steps = b.status()
    assert t == t_end
    got = [x.double().cpu().numpy() for x in st]
    for i, n in enumerate(ncells):
        sl = slice(off[i], off[i + 1])
        z = np.zeros(n)
        q = [u[0][sl], u[1][sl], z, z, u[2][sl], u[3][sl]]
        g = oracle.Grid((n, 1, 1), (1.0 / n, 1.0, 1.0), gamma, (O,) * 6, cfl, rho_mean=float(np.mean(u[0][sl])))
        ref, _, steps_o, _ = oracle.run(g, [a[None, None, :] for a in q], t_end[i])
        assert abs(steps[i] - steps_o) <= 1, (n, steps[i], steps_o)
        for k, f in enumerate((0, 1, 4, 5)):
            e = np.abs(got[k][sl] - ref[f].ravel()).sum()
            assert e <= 1e-4 * max(np.abs(ref[f]).sum(), np.abs(ref[0]).sum() * (1e-3 if f == 1 else 0)), (n, f)
