"""The volume kernel's vector forms: arrays that start on and off 4, 8 and 16
bytes, widths around the lane and tile boundaries, steps of no, one and several
planes.  Every form gives the bits of the aligned call on the same data, writes
nothing outside the volume and keeps NaN, infinities and clamped values."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

U16, F32, F64 = torch.uint16, torch.float32, torch.float64
GEOMETRIES = [(9, 3, 45.0, 0.2, 0.115), (30, 2, 35.0, 0.05, 0.1), (30, 2, 35.0, 0.07, 0.1), (4, 5, 30.0, 0.9, 0.1)]
GUARD = 64


def _bits(t):
    return t.contiguous().view(torch.int16 if t.dtype == U16 else torch.int32 if t.dtype == F32 else torch.int64)


def _off(t, shift):
    """t's values, `shift` elements into a fresh allocation."""
    n = t.numel()
    as_int = _bits(t).reshape(-1)
    buf = torch.zeros(n + shift, dtype=as_int.dtype, device="cuda")
    buf[shift:] = as_int
    return buf[shift:].view(t.dtype).view(t.shape)


def _guarded(shape, dtype, shift):
    n = shape[0] * shape[1] * shape[2]
    ints = {U16: torch.int16, F32: torch.int32, F64: torch.int64}[dtype]
    buf = torch.full((n + 2 * GUARD,), 0x5A5A, dtype=ints, device="cuda")
    lo = GUARD + shift
    return buf, buf[lo:lo + n].view(dtype).view(shape), lo, n


def _raw(shape, dtype, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if dtype == U16:
        return torch.randint(0, 65536, shape, generator=gen, device="cuda", dtype=torch.int32).to(U16)
    raw = torch.randn(shape, generator=gen, device="cuda", dtype=dtype) * 60000.0
    flat = raw.view(-1)
    for i, v in enumerate((float("nan"), float("inf"), -float("inf"), -0.0, 65535.5, 0.5, 1.5)):
        flat[i::97] = v
    return raw


@pytest.mark.parametrize("din,dout", [(U16, F32), (U16, U16), (F32, F32), (F32, U16), (F64, F64)])
@pytest.mark.parametrize("geometry", GEOMETRIES)
def test_every_alignment_gives_the_same_bits(lib, geometry, din, dout):
    for width in (1, 2, 33, 64, 66, 127, 128, 130, 257, 260, 262, 514, 520):
        plan = lib.Plan(geometry[0], geometry[1], width, *geometry[2:])
        raw = _raw(plan.raw_shape, din, width)
        # one column at a time: nothing is a vector there
        one = lib.Plan(geometry[0], geometry[1], 1, *geometry[2:])
        want = lib.deskew(plan, raw, out_dtype=dout)
        for x in {0, width // 2, width - 1}:
            alone = lib.deskew(one, _off(raw[:, :, x:x + 1], 0), out_dtype=dout)
            assert torch.equal(_bits(alone), _bits(want[:, :, x:x + 1])), (width, x)
        for shift, oshift in ((1, 0), (2, 0), (4, 0), (0, 1), (0, 2), (0, 4), (2, 2), (1, 2), (3, 1), (8, 6)):
            buf, vol, lo, n = _guarded(plan.vol_shape, dout, oshift)
            lib.opm_deskew(plan, _off(raw, shift), vol)
            assert torch.equal(_bits(vol), _bits(want)), (width, shift, oshift)
            assert bool((buf[:lo] == 0x5A5A).all()) and bool((buf[lo + n:] == 0x5A5A).all()), (width, shift, oshift)


@pytest.mark.parametrize("din", [U16, F32])
def test_both_volumes_at_every_alignment(lib, din):
    for geometry in GEOMETRIES:
        for width in (2, 66, 127, 130, 260, 262, 520):
            plan = lib.Plan(geometry[0], geometry[1], width, *geometry[2:])
            raw = _raw(plan.raw_shape, din, width)
            want = [lib.deskew(plan, raw, out_dtype=d) for d in (F32, U16)]
            for shift, fshift, hshift in ((0, 0, 0), (1, 0, 0), (2, 2, 2), (0, 2, 4), (0, 4, 2), (0, 1, 0), (3, 0, 1)):
                fbuf, fvol, flo, n = _guarded(plan.vol_shape, F32, fshift)
                hbuf, hvol, hlo, _ = _guarded(plan.vol_shape, U16, hshift)
                lib.opm_deskew_dual(plan, _off(raw, shift), fvol, hvol)
                for got, ref in ((fvol, want[0]), (hvol, want[1])):
                    assert torch.equal(_bits(got), _bits(ref)), (width, shift, fshift, hshift)
                for buf, lo in ((fbuf, flo), (hbuf, hlo)):
                    assert bool((buf[:lo] == 0x5A5A).all()) and bool((buf[lo + n:] == 0x5A5A).all())
