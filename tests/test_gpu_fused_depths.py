"""Volume and live view side by side over the fast kernel's slab depths (its
ring beside a volume is deeper than alone): every output equals the separate
calls', bit for bit."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("ratio", [0.3, 0.45, 0.575, 0.75, 0.95, 1.0])  # 13 to 35 planes a tile row
def test_side_by_side_at_every_ring_depth(lib, ratio):
    plan = lib.Plan(60, 150, 264, 45.0, 0.1 / ratio, 0.1)
    assert lib.opm_plan_path(plan)[0] == lib.OPM_PATH_FAST
    gen = torch.Generator(device="cuda").manual_seed(1)
    raw = torch.randint(0, 65536, plan.raw_shape, generator=gen, device="cuda", dtype=torch.int32).to(torch.uint16)
    want = lib.project(plan, raw, zmip=True, ymip=True)
    for f32, u16 in ((True, False), (False, True), (True, True)):
        for keys in (("zmip",), ("ymip",), ("zmip", "ymip")):
            vf = torch.zeros(plan.vol_shape, device="cuda") if f32 else None
            vu = torch.zeros(plan.vol_shape, dtype=torch.int16, device="cuda").view(torch.uint16) if u16 else None
            out = {k: torch.empty_like(want[k]) for k in keys}
            lib.opm_deskew_mip(plan, raw, vf, vu, **out)
            torch.cuda.synchronize()
            lib.opm_plan_check(plan)
            for k in keys:
                assert torch.equal(out[k], want[k])
            if f32:
                assert torch.equal(vf, lib.deskew(plan, raw))
            if u16:
                ref = lib.deskew(plan, raw, out_dtype=torch.uint16)
                assert torch.equal(vu.view(torch.int16), ref.view(torch.int16))
