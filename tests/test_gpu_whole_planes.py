"""Output columns whose plane coordinate is a whole number, or half of one, on
plans with pixel/step = 1/3 or 1/2 up to rounding.  At 60 and 90 degrees rows
and columns share such coordinates.  A voxel on a plane is that plane's sample,
bit for bit (weight 0, not weight 1 on the plane below, whose FP32 difference
rounds); NEAREST takes the plane the FP64 coordinate is nearest to, where the
ratio is off 1/2 by more than the coordinate's own rounding."""
import numpy as np
import pytest

from oracle import opm as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("theta,cos2", [(60.0, 1), (90.0, 0)])  # 2 cos(theta)
@pytest.mark.parametrize("q,step,pixel", [(3, 0.3, 0.1), (3, 0.345, 0.115), (2, 0.2, 0.1)])
def test_voxels_on_a_plane_are_its_samples(lib, theta, cos2, q, step, pixel):
    plan = lib.Plan(40, 100, 64, theta, step, pixel)
    gen = torch.Generator(device="cuda").manual_seed(q)
    # neighbouring planes of very different size, whose difference rounds
    raw = torch.randn(plan.raw_shape, generator=gen, device="cuda") * 10.0 ** torch.arange(40, device="cuda").remainder(
        5)[:, None, None]
    vol = lib.deskew(plan, raw)
    lib.opm_plan_check(plan)
    num = 2 * (torch.arange(plan.ny, device="cuda") - plan.J0)[None, :] - cos2 * torch.arange(100, device="cuda")[:, None]
    n = torch.div(num, 2 * q, rounding_mode="floor")  # coordinate num / (2 q)
    k, j = torch.nonzero((num % (2 * q) == 0) & (n >= 0) & (n < 40), as_tuple=True)
    assert len(k) > 500
    assert torch.equal(vol[k, j], raw[n[k, j], k])


@pytest.mark.parametrize("theta", [60.0, 90.0])
@pytest.mark.parametrize("off", [4e-15, -4e-15])
def test_nearest_takes_the_nearer_plane_off_the_ratio(lib, theta, off):
    shape = (40, 100, 16, theta, 0.2 * (1.0 + off), 0.1)
    plan = lib.Plan(*shape, interp=1)
    raw = np.arange(40 * 100 * 16).reshape(40, 100, 16).astype(np.uint16)
    vol = lib.deskew(plan, torch.from_numpy(raw.astype(np.int32)).cuda().to(torch.uint16))
    g = O.geometry(*shape)
    # columns whose offset from the tie (off x coordinate) is clear of rounding
    nf = np.abs(O.plane_coord(g, np.arange(g.ny)[None, :], np.zeros((1, 1)))[0])
    j = np.nonzero(nf > 0.4)[0]
    rows = [0] if theta == 60.0 else list(range(100))
    got = vol[rows].cpu().numpy()[:, j]
    want = np.stack([O.deskew_row(raw, g, k, O.NEAREST) for k in rows])[:, j]
    assert np.array_equal(got, want)
