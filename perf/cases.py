"""Workloads of the library as its users call it, for timing and for comparing
results between two versions of the code.

Sizes and geometries are those of the repository's named workloads
(``opm_synth.CONFIGS``, the serving mix, the paper's ROI of 87 x 1304 and 50
frames) and of its tests' ragged shapes.  Stacks hold camera shot noise on a
background of 100 counts with Gaussian blobs of sigma 1.5-4 samples and
200-5000 counts (one per 105,000 samples, as in the live-view workload).

``kind`` names the call: project (live view), deskew (volume), deskew_mip
(volume and live view), skew_grad (forward model and its gradient, one
iteration of the reconstruction), mip_grad (z-MIP and its gradient), batch
(one serving tick), rolling / sliding (a stack arriving frame by frame),
sheet (the paper's sheet-frame view).
"""
import math
import random

import torch

import paper_2211_00645_gb300 as opm
from paper_2211_00645_gb300 import autograd, rolling

BLOB_EVERY = 105_000  # raw samples per blob
BLOB_REACH = 8        # samples a blob extends on each side


def listed():
    live = {"nscan": 200, "nrows": 512, "ncols": 2048, "theta": 35.0, "step": 0.3, "pixel": 0.1}
    diff = {"nscan": 128, "nrows": 256, "ncols": 256, "theta": 30.0, "step": 0.4, "pixel": 0.115}
    paper = {"nscan": 50, "nrows": 87, "ncols": 1304, "theta": 30.0, "step": 0.4, "pixel": 0.115}
    return [
        # the live view of a full acquisition, refreshed once per stack: z- and
        # y-MIP of the headline stack
        {"name": "live_view", "kind": "project", "dtype": "u16", "outs": "zy", **live},
        # the same view at the paper's own ROI (Supp. Fig. 1), where a stack is
        # 11 MB and launches count
        {"name": "live_small", "kind": "project", "dtype": "u16", "outs": "zy", **paper},
        # a camera ROI as a user drags it: nothing is a multiple of anything
        {"name": "live_ragged", "kind": "project", "dtype": "u16", "outs": "zy", "nscan": 151, "nrows": 333,
         "ncols": 1001, "theta": 45.0, "step": 0.2, "pixel": 0.115},
        # widefield-like sum beside the maxima, on the live-view stack
        {"name": "live_sum", "kind": "project", "dtype": "u16", "outs": "zsy", **live},
        # the volume itself, for export and 3-D display
        {"name": "volume_f32", "kind": "deskew", "dtype": "u16", "out": "f32", **live},
        # a large time point stored as uint16, with its live view
        {"name": "volume_large", "kind": "deskew_mip", "dtype": "u16", "out": "u16", "outs": "z", "nscan": 1000,
         "nrows": 1024, "ncols": 2048, "theta": 45.0, "step": 0.2, "pixel": 0.115},
        # one iteration of the gradient-based reconstruction: adjoint and
        # deskew of an FP32 volume through autograd
        {"name": "skew_grad", "kind": "skew_grad", "dtype": "f32", **diff},
        # a loss on the projection: z-MIP forward and its backward, FP32
        {"name": "mip_grad", "kind": "mip_grad", "dtype": "f32", **diff},
        # one tick of the serving loop: six two-channel stacks of uneven ROIs
        {"name": "serving_tick", "kind": "batch", "stacks": 6, "channels": 2, "mix": 5, "theta": 35.0, "step": 0.3,
         "pixel": 0.1},
        # the view refreshed after every exposure at the paper's ROI, frames
        # coming from the camera's pinned host buffers
        {"name": "rolling_small", "kind": "rolling", "frames": "host", **paper},
        # a full-stack view refreshed after every frame of a large ROI
        {"name": "sliding", "kind": "sliding", "frames": "device", "nscan": 50, "nrows": 512, "ncols": 2048,
         "theta": 35.0, "step": 0.3, "pixel": 0.1},
        # the paper's own display: frames shifted by Eq. (1) and maximum-projected
        {"name": "sheet_view", "kind": "sheet", "dtype": "u16", **live},
    ]


def _between(rng, lo, hi):
    """A whole number between lo and hi, spread over the logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _geometry(rng):
    """Sheet angle, scan step and pixel: the named workloads' or any between them."""
    if rng.random() < 0.5:
        t, s, p = rng.choice([(35.0, 0.3, 0.1), (30.0, 0.4, 0.115), (45.0, 0.2, 0.115), (35.0, 0.2, 0.1),
                              (60.0, 0.125, 0.125)])
    else:
        t, s, p = round(rng.uniform(25.0, 60.0), 2), round(rng.uniform(0.12, 0.5), 3), rng.choice([0.1, 0.115])
    return {"theta": t, "step": s, "pixel": p}


def draw(rng):
    kind = rng.choice(["project", "project", "project", "deskew", "deskew_mip", "skew_grad", "mip_grad", "batch",
                       "rolling", "sliding", "sheet"])
    case = {"kind": kind, **_geometry(rng)}
    if kind == "batch":
        case |= {"stacks": rng.randint(1, 6), "channels": rng.choice([1, 2]), "mix": rng.randint(0, 10 ** 6)}
        return case
    nscan, nrows, ncols = _between(rng, 24, 400), _between(rng, 64, 1024), _between(rng, 128, 2048)
    if rng.random() < 0.6:
        ncols = max(128, ncols // 8 * 8)  # cameras offer ROI widths in steps of 8; a crop has any
    if kind in ("project", "deskew", "sheet"):
        case["dtype"] = "u16" if rng.random() < 0.8 else "f32"
    if kind == "project":
        case["outs"] = rng.choice(["z", "zy", "zy", "zs", "zsy"])
    elif kind in ("deskew", "deskew_mip"):
        case["out"] = rng.choice(["f32", "u16"])
        if kind == "deskew_mip":
            case |= {"dtype": "u16", "outs": rng.choice(["z", "zy"])}
    elif kind in ("skew_grad", "mip_grad"):
        nscan, nrows, ncols = _between(rng, 24, 200), _between(rng, 64, 512), _between(rng, 64, 512)
        case["dtype"] = "f32"
    elif kind in ("rolling", "sliding"):
        nscan = _between(rng, 24, 60)
        case["frames"] = rng.choice(["host", "device"])
    case |= {"nscan": nscan, "nrows": nrows, "ncols": ncols}
    while work(case)["bytes"] > 5e9:  # a volume of many columns y': no larger than the live view's
        case["nscan"] = case["nscan"] * 2 // 3
    return case


# ------------------------------------------------------------------- inputs
def _rate(shape, gen):
    """Expected counts: background and blobs, in sixteenths summed as integers
    so that the same seed gives the same stack on every run."""
    n, r, c = shape
    rate = torch.full((n * r * c,), 100 * 16, dtype=torch.int32, device="cuda")
    blobs = max(1, n * r * c // BLOB_EVERY)
    size = torch.tensor([n, r, c], device="cuda")
    centre = torch.rand((blobs, 3), generator=gen, device="cuda", dtype=torch.float64) * size
    sigma = 1.5 + 2.5 * torch.rand(blobs, generator=gen, device="cuda", dtype=torch.float64)
    amp = 200.0 + 4800.0 * torch.rand(blobs, generator=gen, device="cuda", dtype=torch.float64)
    reach = torch.arange(-BLOB_REACH, BLOB_REACH + 1, device="cuda")
    for lo in range(0, blobs, 2000):
        ctr, sig, a = centre[lo:lo + 2000], sigma[lo:lo + 2000], amp[lo:lo + 2000]
        at = ctr.floor().long()[:, :, None] + reach                         # [blob, axis, offset]
        g = torch.exp(-((at - ctr[:, :, None]) / sig[:, None, None]) ** 2 / 2)
        g = torch.where((at >= 0) & (at < size[:, None]), g, 0.0)
        at = at.clamp_(min=0).minimum(size[:, None] - 1)
        val = a[:, None, None, None] * g[:, 0, :, None, None] * g[:, 1, None, :, None] * g[:, 2, None, None, :]
        idx = (at[:, 0, :, None, None] * r + at[:, 1, None, :, None]) * c + at[:, 2, None, None, :]
        rate.index_add_(0, idx.reshape(-1), (val * 16).round().to(torch.int32).reshape(-1))
    return rate.view(n, r, c)


def _stack(shape, seed, dtype="u16"):
    """A camera stack: shot noise (the normal limit of Poisson counts) on _rate."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rate = _rate(shape, gen)
    out = torch.empty(shape, dtype=torch.uint16 if dtype == "u16" else torch.float32, device="cuda")
    for lo in range(0, shape[0], 100):
        lam = rate[lo:lo + 100].float() / 16
        val = torch.randn(lam.shape, generator=gen, device="cuda").mul_(lam.sqrt()).add_(lam)
        if dtype == "u16":
            val.round_().clamp_(0, 65535)
        out[lo:lo + 100] = val.to(out.dtype)
    return out


def _normal(shape, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, generator=gen, device="cuda")


def _shape(case):
    return case["nscan"], case["nrows"], case["ncols"]


def _plan(case, shape=None):
    return opm.Plan(*(shape or _shape(case)), case["theta"], case["step"], case["pixel"])


def _cos(theta):
    return 0.5 if theta == 60.0 else 0.0 if theta == 90.0 else math.cos(math.radians(theta))


def _shear(case):
    """Rows by which a frame is shifted against the one before it (Eq. 1)."""
    return case["step"] * _cos(case["theta"]) / case["pixel"]


def _mix(case):
    """Shapes of a serving tick's stacks: planes, rows and columns per channel."""
    rng = random.Random(case["mix"])
    return [(rng.randrange(50, 401, 50), rng.choice([256, 512, 1024]), rng.choice([512, 1024, 2048]))
            for _ in range(case["stacks"])]


def _empty(*shape):
    return torch.empty(shape, dtype=torch.float32, device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    state = {"case": case, "kind": kind}
    if kind == "batch":
        items, ch = [], case["channels"]
        for i, (n, r, c) in enumerate(_mix(case)):
            plan = _plan(case, (n, r, c))
            raw = _stack((n, r, ch * c), seed * 16 + i)
            for q in range(ch):
                items.append({"plan": plan, "raw": raw[:, :, q * c:], "row_pitch": ch * c, "plane_pitch": r * ch * c,
                              "zmip": _empty(plan.ny, plan.nx), "ymip": _empty(plan.nz, plan.nx)})
        return state | {"items": items, "batch": opm.Batch(len(items), 1 << 18)}
    if kind == "sheet":
        return state | {"raw": _stack(_shape(case), seed, case["dtype"]), "shear": _shear(case)}
    plan = _plan(case)
    state["plan"] = plan
    if kind == "skew_grad":
        state["vol"] = _normal(plan.vol_shape, seed).abs_().mul_(100.0).requires_grad_()
        state["g"] = _normal(plan.raw_shape, seed + 1)
    elif kind == "mip_grad":
        state["raw"] = _stack(_shape(case), seed, "f32").requires_grad_()
        state["g"] = _normal((plan.ny, plan.nx), seed + 1)
    elif kind in ("rolling", "sliding"):
        raw = _stack(_shape(case), seed)
        if case["frames"] == "host":
            host = torch.empty(raw.shape, dtype=torch.uint16, pin_memory=True)
            host.view(torch.int16).copy_(raw.view(torch.int16))
            raw = host
        state["frames"] = list(raw.unbind(0))
        state["view"] = rolling.RollingView(plan, kind)
    else:
        state["raw"] = _stack(_shape(case), seed, case["dtype"])
        if kind == "deskew_mip":
            out = torch.float32 if case["out"] == "f32" else torch.uint16
            state["vol"] = torch.empty(plan.vol_shape, dtype=out, device="cuda")
            state["zmip"] = _empty(plan.ny, plan.nx)
            state["ymip"] = _empty(plan.nz, plan.nx) if "y" in case["outs"] else None
    return state


# ---------------------------------------------------------------------- run
def _signed(t):
    """uint16 counts as int16 bits, which every torch operation takes."""
    return t.view(torch.int16) if t.dtype == torch.uint16 else t


def run(state):
    kind, case = state["kind"], state["case"]
    if kind == "project":
        o = case["outs"]
        return opm.project(state["plan"], state["raw"], zmip="z" in o, zsum="s" in o, ymip="y" in o)
    if kind == "deskew":
        return _signed(opm.deskew(state["plan"], state["raw"],
                                  out_dtype=torch.float32 if case["out"] == "f32" else torch.uint16))
    if kind == "deskew_mip":
        vol = state["vol"]
        f32 = vol.dtype == torch.float32
        opm.opm_deskew_mip(state["plan"], state["raw"], vol_f32=vol if f32 else None, vol_u16=None if f32 else vol,
                           zmip=state["zmip"], ymip=state["ymip"])
        return {"vol": _signed(vol), "zmip": state["zmip"], "ymip": state["ymip"]}
    if kind == "skew_grad":
        state["vol"].grad = None
        raw = autograd.skew(state["vol"], state["plan"])
        raw.backward(state["g"])
        return {"raw": raw.detach(), "grad": state["vol"].grad}
    if kind == "mip_grad":
        state["raw"].grad = None
        z = autograd.zmip(state["raw"], state["plan"])
        z.backward(state["g"])
        return {"zmip": z.detach(), "grad": state["raw"].grad}
    if kind == "batch":
        state["batch"].set(state["items"])
        state["batch"].run(graph=True)
        return [[it["zmip"], it["ymip"]] for it in state["items"]]
    if kind in ("rolling", "sliding"):
        for frame in state["frames"]:
            out = state["view"].push(frame)
        return {"zmip": out["zmip"], "ymip": out["ymip"]}
    return opm.opm_sheet_project(state["raw"], state["shear"])


# --------------------------------------------------------------------- work
def _ny(case, nscan, nrows):
    ratio = case["step"] / case["pixel"]
    j0 = math.ceil(ratio) - 1
    return math.ceil(j0 + nscan * ratio + (nrows - 1) * _cos(case["theta"]) - 1e-9)


def _covered(case, nscan, nrows):
    """Voxels per column x that two planes reach (the others are zero)."""
    return min(nrows * _ny(case, nscan, nrows), round(nrows * (nscan + 1) * case["step"] / case["pixel"]))


def work(case):
    kind = case["kind"]
    if kind == "batch":
        total, flops = 0, 0
        for n, r, c in _mix(case):
            total += case["channels"] * c * (2 * n * r + 4 * _ny(case, n, r) + 4 * r)
            flops += case["channels"] * c * 5 * _covered(case, n, r)
        return {"bytes": total, "flops": flops}
    n, r, c = _shape(case)
    ny, inside = _ny(case, n, r), _covered(case, n, r)
    es = 4 if case.get("dtype") == "f32" else 2
    raw, zmap, ymap, vol = n * r * c, ny * c, r * c, r * ny * c
    if kind == "project":
        o = case["outs"]
        return {"bytes": es * raw + 4 * (zmap * (len(o) - ("y" in o)) + ymap * ("y" in o)),
                "flops": (3 + len(o)) * inside * c}
    if kind in ("deskew", "deskew_mip"):
        out = 4 if case["out"] == "f32" else 2
        mips = 0 if kind == "deskew" else 4 * (zmap + ymap * ("y" in case["outs"]))
        return {"bytes": es * raw + out * vol + mips, "flops": 3 * inside * c}
    if kind == "skew_grad":  # vol -> raw, then g -> grad
        return {"bytes": 4 * (inside * c + raw) + 4 * (raw + vol), "flops": 7 * inside * c}
    if kind == "mip_grad":
        return {"bytes": 4 * (raw + zmap) + 4 * (zmap + raw), "flops": 4 * inside * c + 4 * zmap}
    if kind == "rolling":  # frames in once; each view is updated where its pair reaches
        return {"bytes": 2 * raw + 4 * (zmap + ymap), "flops": 5 * inside * c}
    if kind == "sliding":  # every frame in, every refreshed view out
        return {"bytes": 2 * raw + 4 * n * (zmap + ymap), "flops": 5 * inside * c + 2 * n * (zmap + ymap)}
    rows = r + max(0, math.ceil((n - 1) * _shear(case) - 1e-9))
    return {"bytes": es * raw + 4 * rows * c, "flops": 4 * raw}


# -------------------------------------------------------------------- exact
def _row_weights(case, nscan, nrows, k):
    """Lower plane and weight of every output column j at camera row k."""
    ny = _ny(case, nscan, nrows)
    j = torch.arange(ny, dtype=torch.float64, device="cuda") - (math.ceil(case["step"] / case["pixel"]) - 1)
    nf = (j * case["pixel"] - k * case["pixel"] * _cos(case["theta"])) / case["step"]
    n0 = nf.floor()
    return n0.long(), nf - n0


def _row(case, raw, k):
    """Row k of the deskewed volume, [ny][x], in 64 bits."""
    nscan, nrows, c = raw.shape
    n0, w = _row_weights(case, nscan, nrows, k)
    pad = torch.zeros((nscan + 2, c), dtype=torch.float64, device="cuda")
    pad[1:-1] = _wide(raw[:, k])
    lo, hi = pad[(n0 + 1).clamp(0, nscan + 1)], pad[(n0 + 2).clamp(0, nscan + 1)]
    return lo + w[:, None] * (hi - lo)


def _wide(t):
    return (t.view(torch.int16).to(torch.int32) & 0xFFFF).double() if t.dtype == torch.uint16 else t.double()


def _views(case, raw):
    """z-MIP, its first arg-max, z-sum and y-MIP in 64 bits."""
    nrows = raw.shape[1]
    zm, ym = None, []
    for k in range(nrows):
        v = _row(case, raw, k)
        ym.append(v.amax(0))
        if zm is None:
            zm, zs, az = v.clone(), v.clone(), torch.zeros(v.shape, dtype=torch.int32, device="cuda")
            continue
        az = torch.where(v > zm, k, az)
        zm = torch.maximum(zm, v)
        zs += v
    return zm, az, zs, torch.stack(ym)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out, ch = [], case["channels"]
        for i, (n, r, c) in enumerate(_mix(case)):
            raw = _stack((n, r, ch * c), seed * 16 + i)
            for q in range(ch):
                zm, _, _, ym = _views(case, raw[:, :, q * c:(q + 1) * c].contiguous())
                out.append([zm, ym])
        return out
    shape = _shape(case)
    if kind == "project":
        zm, _, zs, ym = _views(case, _stack(shape, seed, case["dtype"]))
        o = case["outs"]
        return {k: v for k, v, on in (("zmip", zm, "z"), ("zsum", zs, "s"), ("ymip", ym, "y")) if on in o}
    if kind in ("rolling", "sliding"):
        zm, _, _, ym = _views(case, _stack(shape, seed))
        return {"zmip": zm, "ymip": ym}
    if kind in ("deskew", "deskew_mip"):
        raw = _stack(shape, seed, case["dtype"])
        vol = None
        if case["out"] == "f32":
            vol = torch.stack([_row(case, raw, k) for k in range(shape[1])])
        if kind == "deskew":
            return vol
        zm, _, _, ym = _views(case, raw)
        return {"vol": vol, "zmip": zm, "ymip": ym if "y" in case["outs"] else None}
    if kind == "sheet":
        raw = _stack(shape, seed, case["dtype"])
        n, r, c = shape
        rows = r + max(0, math.ceil((n - 1) * _shear(case) - 1e-9))
        y = torch.arange(rows, dtype=torch.float64, device="cuda")
        out = torch.zeros((rows, c), dtype=torch.float64, device="cuda")
        for q in range(n):
            at = y - q * _shear(case)
            lo = at.floor()
            pad = torch.zeros((r + 2, c), dtype=torch.float64, device="cuda")
            pad[1:-1] = _wide(raw[q])
            lo_i = (lo.long() + 1).clamp(0, r + 1)
            hi_i = (lo.long() + 2).clamp(0, r + 1)
            v = pad[lo_i] + (at - lo)[:, None] * (pad[hi_i] - pad[lo_i])
            out = v if q == 0 else torch.maximum(out, v)
        return out
    nscan, nrows, c = shape
    ny = _ny(case, nscan, nrows)
    planes = torch.arange(nscan, dtype=torch.float64, device="cuda")[:, None]
    if kind == "skew_grad":
        vol, g = _normal((nrows, ny, c), seed).abs_().mul_(100.0), _normal(shape, seed + 1)
    else:
        raw = _stack(shape, seed, "f32")
        zm, az, _, _ = _views(case, raw)
        g = _normal((ny, c), seed + 1).double()
    rows, grad = [], []
    for k in range(nrows):
        n0, w = _row_weights(case, nscan, nrows, k)
        tent = (1 - ((n0 + w)[None, :] - planes).abs()).clamp(min=0)  # [nscan][ny]
        if kind == "skew_grad":
            rows.append(tent @ vol[k].double())
            grad.append(tent.T @ g[:, k].double())
        else:
            grad.append(tent @ torch.where(az == k, g, 0.0))
    if kind == "skew_grad":
        return {"raw": torch.stack(rows, 1), "grad": torch.stack(grad)}
    return {"zmip": zm, "grad": torch.stack(grad, 1)}
