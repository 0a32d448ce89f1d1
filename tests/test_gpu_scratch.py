"""A handle's scratch: what it holds on the device, and the FP32 steps that share or cut it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1607_01105_gb300 import inputs, ppml  # noqa: E402

pytestmark = pytest.mark.gpu

F32, F64 = ppml.PPML_F32, ppml.PPML_F64
O, P = ppml.OUTFLOW, ppml.PERIODIC


def _held(n, dtype):
    """Bytes a handle of the grid takes on the device, beyond what the caller holds."""
    u = [torch.ones(int(np.prod(n)), device="cuda", dtype=ppml.torch_dtype(dtype)) for _ in range(6)]
    small = [x[:4096] for x in u]
    ppml.Grid((16, 16, 16), (1.0,) * 3, 1.4, 0.2, (O,) * 6, dtype, u0=small).close()  # (modules loaded)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    grid = ppml.Grid(n, (1.0,) * 3, 1.4, 0.2, (O,) * 6, dtype, u0=u)
    held = before - torch.cuda.mem_get_info()[0]
    grid.close()
    return held


@pytest.mark.parametrize("dtype,per_cell", [(F32, 36), (F64, 40)])
@pytest.mark.parametrize("n", [(256, 256, 256), (512, 512, 64)])
def test_handle_holds_no_more_than_the_intermediate_state(n, dtype, per_cell):
    """U* (five fields, in FP32 and four low parts), and a few MB of partials and rounding."""
    assert _held(n, dtype) <= per_cell * int(np.prod(n)) + (16 << 20)


@pytest.mark.parametrize("n", [(130, 130, 130), (4096, 2048, 3)])
def test_handle_of_padded_tiles_is_bounded(n):
    """Grids whose tiles are mostly padding: 256 MB for the low parts' space at most."""
    assert _held(n, F32) <= 20 * int(np.prod(n)) + max(256 << 20, 16 * int(np.prod(n))) + (16 << 20)


def _fields(n, seed):
    pb = inputs.random_smooth(n=n, bc=(P,) * 6)
    return [np.roll(a, seed, axis=2) for a in pb.u]


def test_fp32_step_in_several_launches_of_a_handle():
    """5292 tiles, mostly padding, of which the face velocities hold 5140: two launches.  The
    state repeats along x, so each half has the bits of the grid of one period (2646 tiles)."""
    n = (672, 1008, 3)
    one = ppml.to_device(_fields(n, 0), F32)
    two = [torch.cat([a.view(3, 1008, 672)] * 2, dim=2).reshape(-1).contiguous() for a in one]
    out = []
    for m, u in ((n, one), ((1344, 1008, 3), two)):
        grid = ppml.Grid(m, (0.01,) * 3, 1.4, 0.2, (P,) * 6, F32, u0=u)
        a, b = [torch.empty_like(x) for x in u], [torch.empty_like(x) for x in u]
        grid.step(u, a, 5e-4)
        grid.step(a, b, 5e-4)
        out.append((b, grid.diag()))
    for f in range(6):
        small, big = out[0][0][f].view(3, 1008, 672), out[1][0][f].view(3, 1008, 1344)
        assert torch.equal(big[:, :, :672], small) and torch.equal(big[:, :, 672:], small), f
    assert out[0][1]["vmax"] == out[1][1]["vmax"] and out[0][1]["cmax"] == out[1][1]["cmax"]


def test_plain_and_double_float_steps_share_a_handle():
    """The two kinds of FP32 step alternate on one handle, whose low parts and face velocities
    share their space: the bits of handles of their own."""
    n = (33, 40, 35)
    hi = ppml.to_device(_fields(n, 0), F32)
    pair = hi + [1e-9 * x for x in hi[:5]]

    def grid(u):
        return ppml.Grid(n, (0.02,) * 3, 1.4, 0.2, (P,) * 6, F32, u0=u)

    def steps(g, u, count):
        for _ in range(count):
            v = [torch.empty_like(x) for x in u]
            g.step(u, v, 1e-3)
            u = v
        return u

    plain, double = steps(grid(hi), hi, 3), steps(grid(pair), pair, 3)
    g = grid(hi)
    a, b = hi, pair
    for _ in range(3):
        a, b = steps(g, a, 1), steps(g, b, 1)
    assert all(torch.equal(x, y) for x, y in zip(a + b, plain + double))


@pytest.mark.parametrize("n,launches", [((3, 3, 29127), 12), ((17, 17, 907), 2), ((64, 64, 64), 1),
                                        ((16, 16, 16 * 64), 1), ((3, 3, 3), 1)])
def test_noalloc_step_uses_the_whole_buffer(n, launches):
    """The allocation-free FP32 step: as many tiles a launch as its buffer holds, and the bits
    of the handle's step."""
    from torch.profiler import ProfilerActivity, profile
    u = ppml.to_device(inputs.random_smooth(n=n, bc=(P,) * 6).u, F32)
    a, b = [torch.empty_like(x) for x in u], [torch.empty_like(x) for x in u]
    h, rho = (0.02,) * 3, float(u[0].double().mean())
    grid = ppml.Grid(n, h, 1.4, 0.2, (P,) * 6, F32, u0=u, rho_ref=rho)
    grid.step(u, a, 1e-3)
    desc = ppml.make_desc(n, h, 1.4, 0.2, (P,) * 6, F32)
    for _ in range(3):  # (a process's first session may record nothing)
        torch.cuda.synchronize()
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            out = ppml.step_noalloc(desc, u, b, 1e-3, rho)
            torch.cuda.synchronize()
        count = sum(e.count for e in prof.key_averages() if "face_velocity" in e.key)
        if count:
            break
    assert all(torch.equal(x, y) for x, y in zip(a, b))
    d = grid.diag()
    assert out[0] == d["dt_next"] and out[3] == d["sums"]
    if not count:
        pytest.skip("the profiler records no kernels here")
    assert count == launches
