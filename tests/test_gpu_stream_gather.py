"""The gathering plane-pair and sliding kernels where their runs and vectors
end: odd widths, frames off 8 bytes, runs that skip rows or columns (steep
shears, pixel > step), 90 degrees (one run per column), few rows.  All pairs
together equal opm_project bit for bit; the z-sum of nz FP32 terms is within
nz 2^-24 sum V of the exact sum, the bound of recursive summation."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

GEOMETRIES = [
    (11, 40, 35.0, 0.3, 0.1),
    (9, 33, 90.0, 0.125, 0.125),
    (8, 70, 20.0, 0.1, 0.09),
    (12, 21, 30.0, 0.05, 0.2),    # pixel = 4 steps: pairs without a column in some rows
    (2, 1, 45.0, 0.2, 0.115),
    (6, 300, 60.0, 0.5, 0.1),
]


def _stack(shape, shift, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n = shape[0] * shape[1] * shape[2]
    return torch.randint(0, 65536, (n + shift,), generator=gen, device="cuda", dtype=torch.int32).to(
        torch.uint16)[shift:].view(shape)


@pytest.mark.parametrize("width,shift", [(1, 0), (37, 3), (128, 0), (132, 4), (133, 0), (260, 1)])
@pytest.mark.parametrize("geometry", GEOMETRIES)
def test_all_pairs_and_pushes_equal_the_projection(lib, geometry, width, shift):
    plan = lib.Plan(geometry[0], geometry[1], width, *geometry[2:])
    raw = _stack(plan.raw_shape, shift, width)
    want = lib.project(plan, raw, zmip=True, zsum=True, ymip=True)
    z, s = torch.empty(2, plan.ny, plan.nx, device="cuda")
    y = torch.empty(plan.nz, plan.nx, device="cuda")
    lib.opm_stream_begin(plan, z, s, y)
    for n in range(-1, plan.nscan):
        lo = raw[n] if n >= 0 else None
        hi = raw[n + 1] if n + 1 < plan.nscan else None
        lib.opm_stream_pair(plan, lo, hi, n, z, s, y)
    # the sliding view over two different stacks, checked after every push
    per = (plan.ny + plan.nz) * plan.nx
    run, view, slots = (torch.zeros(k, device="cuda") for k in (per, per, plan.nscan * per))
    slots = slots.view(plan.nscan, per)
    stack = torch.zeros(raw.numel() + shift, dtype=torch.int16, device="cuda").view(torch.uint16)[shift:].view(raw.shape)
    for source in (raw, _stack(plan.raw_shape, 0, width + 1)):
        for m in range(plan.nscan):
            stack[m].view(torch.int16).copy_(source[m].view(torch.int16))
            lib.opm_sliding_push(plan, stack, m, run, slots, view)
            now = lib.project(plan, stack, zmip=True, ymip=True)
            assert torch.equal(view[:plan.ny * plan.nx].view(plan.ny, plan.nx), now["zmip"]), m
            assert torch.equal(view[plan.ny * plan.nx:].view(plan.nz, plan.nx), now["ymip"]), m
    lib.opm_plan_check(plan)
    assert torch.equal(z, want["zmip"]) and torch.equal(y, want["ymip"])
    exact = lib.deskew(plan, raw).double().sum(0)
    bound = plan.nz * 2.0 ** -24 * exact
    assert bool(((s.double() - exact).abs() <= bound).all())
