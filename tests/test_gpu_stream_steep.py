"""Plane pairs and sliding pushes whose columns are shared by several warps:
long runs of rows (steep sheets, small pixel / step, 90 degrees) on few columns,
runs that do not divide among the warps, rows on and off 8 bytes.  All pairs
together, and every push, equal opm_project bit for bit; the z-sum of nz FP32
terms is within nz 2^-24 sum V of the exact sum and the same on every run."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

GEOMETRIES = [
    (5, 300, 90.0, 0.125, 0.125),  # one column per pair: 16 warps on every width
    (4, 517, 90.0, 0.3, 0.1),
    (6, 300, 89.0, 0.3, 0.1),      # 172 rows a run: 16 warps, 8 on the widest
    (4, 90, 88.0, 0.5, 0.1),       # the whole column
    (8, 131, 85.0, 0.3, 0.1),      # 34 rows: 4 warps
    (7, 97, 75.0, 0.2, 0.115),     # 7 rows: 4 warps or 1
]


def _stack(shape, shift, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n = shape[0] * shape[1] * shape[2]
    return torch.randint(0, 65536, (n + shift,), generator=gen, device="cuda", dtype=torch.int32).to(
        torch.uint16)[shift:].view(shape)


@pytest.mark.parametrize("width,shift", [(3, 0), (36, 4), (133, 1), (260, 0), (2056, 0), (2051, 0)])
@pytest.mark.parametrize("geometry", GEOMETRIES)
@pytest.mark.parametrize("interp", [0, 1])
def test_shared_columns_equal_the_projection(lib, geometry, width, shift, interp):
    plan = lib.Plan(geometry[0], geometry[1], width, *geometry[2:], interp=interp)
    raw = _stack(plan.raw_shape, shift, width)
    want = lib.project(plan, raw, zmip=True, ymip=True)
    sums = []
    for _ in range(2):
        z, s = torch.empty(2, plan.ny, plan.nx, device="cuda")
        y = torch.empty(plan.nz, plan.nx, device="cuda")
        lib.opm_stream_begin(plan, z, s, y)
        for n in range(-1, plan.nscan):
            lo = raw[n] if n >= 0 else None
            hi = raw[n + 1] if n + 1 < plan.nscan else None
            lib.opm_stream_pair(plan, lo, hi, n, z, s, y)
        sums.append(s)
        assert torch.equal(z, want["zmip"]) and torch.equal(y, want["ymip"])
    exact = lib.deskew(plan, raw).double().sum(0)
    assert bool(((sums[0].double() - exact).abs() <= plan.nz * 2.0 ** -24 * exact).all())
    assert torch.equal(sums[0], sums[1])
    # z-MIP alone (no rows), and the sliding view over two stacks
    z1 = torch.zeros(plan.ny, plan.nx, device="cuda")
    for n in range(-1, plan.nscan):
        lib.opm_stream_pair(plan, raw[n] if n >= 0 else None, raw[n + 1] if n + 1 < plan.nscan else None, n, z1)
    assert torch.equal(z1, want["zmip"])
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
