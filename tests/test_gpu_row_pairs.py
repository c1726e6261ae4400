"""Row pairs of the periodic kernel: bands with one row or an odd number of
rows of a phase, units that end inside a phase, odd unit lengths in a batch
(rounded up to whole pairs), and pixel/step written in ways that are not the
compiled ratio to the last bit.  The maxima are the volume's, bit for bit."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = [
    ((30, 1, 128, 35.0, 0.3, 0.1), (1, 3)),
    ((30, 2, 136, 35.0, 0.3, 0.1), (1, 3)),
    ((17, 61, 200, 47.0, 0.345, 0.115), (1, 3)),
    ((40, 90, 264, 25.0, 0.45, 0.15), (1, 3)),
    ((90, 37, 128, 89.0, 0.2, 0.1), (1, 2)),     # hardly any shift from row to row: one phase
    ((45, 64, 160, 31.0, 0.23, 0.115), (1, 2)),
]


@pytest.mark.parametrize("interp", [0, 1])
@pytest.mark.parametrize("shape,pq", CASES)
def test_paired_rows_match_the_volume(lib, shape, pq, interp):
    plan = lib.Plan(*shape, interp=interp)
    assert lib.opm_plan_path(plan) == (lib.OPM_PATH_PERIODIC, *pq)
    gen = torch.Generator(device="cuda").manual_seed(shape[1])
    raw = torch.randint(0, 65536, plan.raw_shape, generator=gen, device="cuda", dtype=torch.int32).to(torch.uint16)
    vol = lib.deskew(plan, raw)
    both = lib.project(plan, raw, zmip=True, ymip=True)
    z_only = lib.project(plan, raw, zmip=True)
    batch = lib.Batch(max_items=1)
    torch.cuda.synchronize()
    lib.opm_plan_check(plan)
    assert torch.equal(both["zmip"], vol.amax(0)) and torch.equal(both["ymip"], vol.amax(1))
    assert torch.equal(z_only["zmip"], vol.amax(0))
    item = {"plan": plan, "raw": raw, "zmip": torch.empty_like(both["zmip"]), "ymip": torch.empty_like(both["ymip"])}
    for kchunk in (0, 1, 7, 64, 1000):
        for shape_id in (lib.OPM_SHAPE_PER_J32X2, lib.OPM_SHAPE_PER_J16X2, lib.OPM_SHAPE_FAST_J8X4):
            item["zmip"].fill_(-1)
            item["ymip"].fill_(-1)
            batch.set([item], kchunk, shape_id)
            batch.run()
            torch.cuda.synchronize()
            batch.check()
            assert torch.equal(item["zmip"], both["zmip"]) and torch.equal(item["ymip"], both["ymip"]), (kchunk, shape_id)
    batch.close()
