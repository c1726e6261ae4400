"""Capacity of a batch's work list with periodic and general items together:
the list that just holds the rows in order (one unit per 32-column tile, row
chunk and x-tile, and one per tile of the general items) holds the row pairs
too.  64 rows make 33 pairs here where two phases have an odd number of rows."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _items(lib, outs):
    items = []
    for keys in outs:
        plan = lib.Plan(120, 64, 256, 35.0, 0.3, 0.1)
        gen = torch.Generator(device="cuda").manual_seed(len(items))
        raw = torch.randint(0, 65536, plan.raw_shape, generator=gen, device="cuda", dtype=torch.int32).to(torch.uint16)
        size = {"zmip": (plan.ny, plan.nx), "zsum": (plan.ny, plan.nx), "ymip": (plan.nz, plan.nx)}
        items.append({"plan": plan, "raw": raw, **{k: torch.empty(size[k], device="cuda") for k in keys}})
    return items


@pytest.mark.parametrize("kchunk", [16, 32, 64])
def test_row_pairs_leave_room_for_general_items(lib, kchunk):
    fast, general = ["zmip", "ymip"], ["zmip", "zsum", "ymip"]
    items = _items(lib, [fast, fast] + [general] * 3)
    plan = items[0]["plan"]
    big = lib.Batch(5)
    big.set(items[:2], kchunk, lib.OPM_SHAPE_FAST_J8X4)  # rows in order
    room = big.info()["units"] + 3 * ((plan.ny + 31) // 32) * (plan.nx // 128)
    want = [lib.project(it["plan"], it["raw"], zmip=True, zsum=True, ymip=True) for it in items]
    tight = lib.Batch(5, room)
    tight.set(items, kchunk)
    tight.run()
    torch.cuda.synchronize()
    tight.check()
    assert tight.info()["units"] <= room and tight.info()["shape"] == lib.OPM_SHAPE_PER_J32X2
    for it, ref in zip(items, want):
        for key in ("zmip", "zsum", "ymip"):
            if key in it:
                assert torch.equal(it[key], ref[key]), key
