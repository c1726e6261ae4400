"""The direct projection kernel over its tilings: 8, 4 and 2 warps to a tile's
rows, several tiles per CTA (y-maxima and partial results meet in shared memory),
tiles past the grid's last column, both ways of keeping arg-max rows, and values
that are no numbers.  Reference: the deskewed volume.  Maxima and arg-max rows are
its bits; a z-sum of nz FP32 terms in any order is within nz 2^-24 sum|V| of their
exact sum."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# (warps per tile, width, geometry): the fewest of 2, 4, 8 that make 2432 warps over
# ceil(ny / 8) x ceil(width / 128) tiles.  ny off 8, 16 and 32, rows off 32, widths
# on and off the vectors.
SHAPES = [
    (8, 520, (24, 40, 45.0, 0.2, 0.115)),
    (4, 8712, (24, 40, 45.0, 0.2, 0.115)),
    (4, 9001, (23, 37, 45.0, 0.2, 0.115)),
    (2, 17416, (24, 40, 45.0, 0.2, 0.115)),
    (2, 17402, (21, 33, 35.0, 0.3, 0.1)),
    (2, 65540, (3, 70, 35.0, 0.3, 0.1)),
    (4, 78001, (9, 3, 35.0, 0.05, 0.1)),
    (2, 65539, (30, 5, 60.0, 0.07, 0.1)),
]


def _tiles(plan):
    return -(-plan.ny // 8) * -(-plan.nx // 128)


def _raw(plan, dtype, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    vals = torch.randint(0, 4000, plan.raw_shape, generator=gen, device="cuda", dtype=torch.int32)
    return vals.to(torch.uint16) if dtype == torch.uint16 else vals.float() * 0.37 - 500.0


def _reference(vol):
    zmip, ymip = vol.amax(0), vol.amax(1)
    return {"zmip": zmip, "ymip": ymip, "argz": (vol == zmip).to(torch.int8).argmax(0).to(torch.int32)}


def _check(out, ref, vol):
    for key, val in out.items():
        if key == "zsum":
            bound = vol.shape[0] * 2.0 ** -24 * vol.abs().sum(0, dtype=torch.float64)
            assert bool(((val.double() - vol.sum(0, dtype=torch.float64)).abs() <= bound).all())
        else:
            assert torch.equal(val, ref[key]), key


@pytest.mark.parametrize("dtype", ["uint16", "float32"])
@pytest.mark.parametrize("warps,width,geometry", SHAPES)
def test_every_tiling_matches_the_volume(lib, warps, width, geometry, dtype):
    plan = lib.Plan(geometry[0], geometry[1], width, *geometry[2:])
    assert next((w for w in (2, 4) if _tiles(plan) * w >= 16 * 152), 8) == warps
    raw = _raw(plan, getattr(torch, dtype), width)
    vol = lib.deskew(plan, raw)
    ref = _reference(vol)
    alls = lib.project(plan, raw, zmip=True, zsum=True, ymip=True, argz=True)
    sums = lib.project(plan, raw, zmip=False, zsum=True)
    _check(alls, ref, vol)
    _check(sums, ref, vol)
    assert torch.equal(alls["zsum"], sums["zsum"])
    _check(lib.project(plan, raw, zmip=False, zsum=True, ymip=True), ref, vol)
    _check(lib.project(plan, raw, zmip=True, ymip=True, argz=True), ref, vol)
    _check(lib.project(plan, raw, zmip=False, ymip=True, argz=False), ref, vol)
    lib.opm_plan_check(plan)
    if dtype != "uint16" or width % 8:
        return
    # the same in a batch: single pieces, and whole 32-column tiles where the list
    # has no room for pieces; beside another item the groups differ
    jtiles, xtiles = -(-plan.ny // 32), -(-plan.nx // 128)
    for units, count in ((1 << 20, 1), (1 << 20, 2), (jtiles * xtiles, 1)):
        for keys in (("zmip", "ymip"), ("zmip", "zsum", "ymip", "argz"), ("argz",), ("zsum", "ymip")):
            items = [{"plan": plan, "raw": raw, **{k: torch.full_like(alls[k], -7) for k in keys}} for _ in range(count)]
            batch = lib.Batch(count, units)
            batch.set(items, 0, lib.OPM_SHAPE_GEN_J8X4)
            batch.run()
            torch.cuda.synchronize()
            batch.check()
            for it in items:
                for k in keys:
                    assert torch.equal(it[k], alls[k]), (k, units, count)
            batch.close()


@pytest.mark.parametrize("nrows", [65534, 65535, 65536, 65537])
def test_arg_max_rows_past_16_bits(lib, nrows):
    """All outputs keep the rows in 16 bits up to 65535 rows: maxima in the first
    and the last row, in none (all zero), and ties that the first row wins."""
    plan = lib.Plan(2, nrows, 6, 90.0, 0.1, 0.1)
    for dtype in (torch.uint16, torch.float32):
        raw = torch.zeros(plan.raw_shape, dtype=torch.int32, device="cuda")
        raw[:, nrows - 1, 1] = 9
        raw[:, 0, 2] = 5
        raw[:, nrows - 2, 3] = 7
        raw[:, 40000:, 4] = 3
        raw[0, :, 5] = torch.arange(nrows, device="cuda") % 60000
        raw = raw.to(dtype)
        vol = lib.deskew(plan, raw)
        out = lib.project(plan, raw, zmip=True, zsum=True, ymip=True, argz=True)
        _check(out, _reference(vol), vol)
        _check(lib.project(plan, raw, zmip=True, argz=True), _reference(vol), vol)


@pytest.mark.parametrize("width", [132, 133, 17416])
def test_nan_and_infinities(lib, width):
    """Maxima pass NaN over (a column of nothing else is -inf, row 0); the z-sum is
    NaN or infinite where the volume's is."""
    plan = lib.Plan(12, 45, width, 45.0, 0.2, 0.115)
    raw = _raw(plan, torch.float32, width)
    flat = raw.view(-1)
    for i, v in enumerate((float("nan"), float("inf"), -float("inf"))):
        flat[13 * i::131] = v
    raw[:, :, 7] = float("nan")
    vol = lib.deskew(plan, raw)
    low = torch.where(vol.isnan(), torch.tensor(-float("inf"), device="cuda"), vol)
    ref = _reference(low)
    ref["argz"] = torch.where(ref["zmip"] == -float("inf"), torch.zeros_like(ref["argz"]), ref["argz"])
    for keys in (("zmip", "ymip"), ("zmip", "argz"), ("zmip", "zsum", "ymip", "argz")):
        out = lib.project(plan, raw, **{k: k in keys for k in ("zmip", "zsum", "ymip", "argz")})
        for k in keys:
            if k == "zsum":
                want = vol.sum(0)
                assert torch.equal(out[k].isnan(), want.isnan()) and torch.equal(out[k].isinf(), want.isinf())
            else:
                assert torch.equal(out[k], ref[k]), k
