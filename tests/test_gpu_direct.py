"""The direct projection kernel (z-sum, arg-max, FP32 input, rows of any width
and alignment, any plane step): against the deskewed volume of the volume
kernel.  Maxima and arg-max rows are the volume's bit for bit.  A z-sum of nz
FP32 terms in any order is within nz 2^-24 sum|V| of the exact sum of those
terms, the usual bound of recursive summation."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# (nscan, nrows, theta, step, pixel): column steps of 1/3, 0.575 and 1 plane
# and of several planes; few columns (ny < 32), column counts off the 8- and
# 32-column tiles, fewer rows than row groups
GEOMETRIES = [
    (21, 45, 35.0, 0.3, 0.1),
    (24, 37, 45.0, 0.2, 0.115),
    (17, 70, 60.0, 0.125, 0.125),
    (20, 33, 35.0, 0.05, 0.1),
    (9, 3, 30.0, 0.1, 0.35),
    (40, 5, 20.0, 0.4, 0.115),
]
# widths around the 128-column tile and vector boundaries, with the stack
# starting `shift` elements into its allocation
WIDTHS = [(1, 0), (7, 3), (64, 0), (127, 1), (128, 0), (129, 2), (132, 4), (260, 0), (301, 5)]


def _raw(shape, width, shift, dtype, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n = shape[0] * shape[1] * width
    vals = torch.randint(0, 4000, (n + shift,), generator=gen, device="cuda").float()
    if dtype == torch.float32:
        vals = vals * 0.37 - 500.0
    return vals.to(dtype)[shift:].view(shape[0], shape[1], width)


@pytest.mark.parametrize("dtype", ["uint16", "float32"])
@pytest.mark.parametrize("geometry", GEOMETRIES)
def test_direct_outputs_match_the_volume(lib, geometry, dtype):
    dtype = getattr(torch, dtype)
    for width, shift in WIDTHS:
        raw = _raw(geometry[:2], width, shift, dtype, width)
        plan = lib.Plan(geometry[0], geometry[1], width, *geometry[2:])
        vol = lib.deskew(plan, raw)
        alls = lib.project(plan, raw, zmip=True, zsum=True, ymip=True, argz=True)
        sums = lib.project(plan, raw, zmip=True, zsum=True)
        args = lib.project(plan, raw, zmip=False, ymip=True, argz=True)
        maxs = lib.project(plan, raw, zmip=True, ymip=True)
        torch.cuda.synchronize()
        lib.opm_plan_check(plan)
        zmip, ymip = vol.amax(0), vol.amax(1)
        first = (vol == zmip).to(torch.int32).argmax(0).to(torch.int32)
        for out in (alls, sums, args, maxs):
            for key, want in (("zmip", zmip), ("ymip", ymip), ("argz", first)):
                if key in out:
                    assert torch.equal(out[key], want), (key, width, shift)
        bound = plan.nz * 2.0 ** -24 * vol.double().abs().sum(0)
        exact = vol.double().sum(0)
        for out in (alls, sums):
            assert bool(((out["zsum"].double() - exact).abs() <= bound).all()), (width, shift)
        assert torch.equal(alls["zsum"], sums["zsum"])


def test_direct_reads_only_the_stack(lib):
    """Chunks that reach past the stack's ends leave its neighbours out: the
    values around an unaligned stack do not show in any output."""
    nscan, nrows, width = 9, 7, 43
    plan = lib.Plan(nscan, nrows, width, 45.0, 0.2, 0.115)
    n = nscan * nrows * width
    for shift in range(8):
        got = []
        for fill in (0, 65535):
            buf = torch.full((n + 32,), fill, dtype=torch.int32, device="cuda").to(torch.uint16)
            raw = buf[8 + shift:8 + shift + n].view(nscan, nrows, width)
            raw.view(torch.int16).copy_((torch.arange(n, device="cuda") % 777).to(torch.int16).view(nscan, nrows, width))
            got.append(lib.project(plan, raw, zmip=True, zsum=True, ymip=True, argz=True))
        torch.cuda.synchronize()
        for key in got[0]:
            assert torch.equal(got[0][key], got[1][key]), (key, shift)
