"""Periodic plans whose weights do not repeat (pixel/step a little above the
compiled ratio) beside ones whose weights do: maxima against the volume's, bit
for bit, alone, in one batch, and in a captured batch launch."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SHAPES = [(50, 87, 264, 30.0), (30, 20, 136, 45.0), (17, 61, 128, 47.0)]


def _item(lib, shape, q, off, interp):
    plan = lib.Plan(*shape, 0.1 * q * (1.0 - off), 0.1, interp=interp)
    assert lib.opm_plan_path(plan) == (lib.OPM_PATH_PERIODIC, 1, q)
    gen = torch.Generator(device="cuda").manual_seed(shape[1])
    raw = torch.randint(0, 65536, plan.raw_shape, generator=gen, device="cuda", dtype=torch.int32).to(torch.uint16)
    vol = lib.deskew(plan, raw)
    return {"plan": plan, "raw": raw, "zmip": torch.empty((plan.ny, plan.nx), device="cuda"),
            "ymip": torch.empty((plan.nz, plan.nx), device="cuda")}, vol.amax(0), vol.amax(1)


@pytest.mark.parametrize("q,interp", [(3, 0), (3, 1), (2, 0)])
@pytest.mark.parametrize("off", [1e-11, 1e-6, 1e-5])
def test_weights_of_every_column(lib, q, off, interp):
    got = [_item(lib, s, q, o, interp) for s in SHAPES for o in (off, 0.0)]
    for it, zmip, ymip in got:
        both = lib.project(it["plan"], it["raw"], zmip=True, ymip=True)
        z_only = lib.project(it["plan"], it["raw"], zmip=True)
        lib.opm_plan_check(it["plan"])
        assert torch.equal(both["zmip"], zmip) and torch.equal(both["ymip"], ymip) and torch.equal(z_only["zmip"], zmip)
    batch = lib.Batch(len(got))
    for shape_id in (lib.OPM_SHAPE_PER_J32X2, lib.OPM_SHAPE_PER_J16X2):
        # repeating weights alone, then with the others in the same launch shape
        for items in (got[1::2], got, got[1::2]):
            for it, _, _ in items:
                it["zmip"].fill_(-1)
                it["ymip"].fill_(-1)
            batch.set([it for it, _, _ in items], 0, shape_id)
            batch.run(graph=True)
            torch.cuda.synchronize()
            batch.check()
            for it, zmip, ymip in items:
                assert torch.equal(it["zmip"], zmip) and torch.equal(it["ymip"], ymip)
    batch.close()
