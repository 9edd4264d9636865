"""Performance cases: the work that users of this package have it do, through
its public entry points (DegridPlan.degrid and .grid, DegridFn,
SubgridPredictor.predict, pack_subgrids).

Values and distributions are those of the repository's workloads: complex
Gaussian subgrids, visibilities on straight lines (the usual test of the
method), on unions of lines and circular arcs with uneven counts, or
scattered over the subgrid, Kaiser-Bessel kernels, a model sky of point
sources.  Everything is made on the GPU from the seed.  `exact` is the
definition in 64-bit torch and shares no code with the package.
"""
import functools
import math

import numpy as np
import torch

import paper_2102_12739_gb300 as dg

UV_SUPPORT, W_SUPPORT = 8, 4
UV_OVERSAMPLE, W_OVERSAMPLE = 16384, 128
DEVICE = "cuda"


# ---- the cases -------------------------------------------------------------

def listed():
    return [
        # an interactive or streaming call: one subgrid, one short track; the
        # launches and latencies of a call are what it costs
        {"name": "degrid_line_20k", "kind": "degrid", "list": "line", "S": 1, "n": 20000, "uneven": False,
         "ny": 512, "nx": 512, "nz": 4, "dtype": "c64", "table": "1d", "gather": False, "comp": False},
        # predicting a whole observation: long dense tracks over a stack of subgrids
        {"name": "degrid_lines_16m", "kind": "degrid", "list": "line", "S": 64, "n": 16000000, "uneven": False,
         "ny": 512, "nx": 512, "nz": 4, "dtype": "c64", "table": "1d", "gather": False, "comp": False},
        # the same with 16-bit storage, track pieces of very uneven length per
        # subgrid (counts log-uniform over three decades)
        {"name": "degrid_uneven_bf16", "kind": "degrid", "list": "pieces", "S": 96, "n": 14000000, "uneven": True,
         "ny": 512, "nx": 512, "nz": 4, "dtype": "bf16", "table": "1d", "gather": False, "comp": False},
        # sparse coverage: no two neighbours share a footprint
        {"name": "degrid_scatter_c64", "kind": "degrid", "list": "scatter", "S": 16, "n": 4000000, "uneven": False,
         "ny": 512, "nx": 512, "nz": 4, "dtype": "c64", "table": "1d", "gather": True, "comp": False},
        # sparse coverage, 16-bit storage, compensated sums, ragged sizes
        {"name": "degrid_scatter_f16", "kind": "degrid", "list": "scatter", "S": 13, "n": 1234567, "uneven": True,
         "ny": 500, "nx": 488, "nz": 4, "dtype": "f16", "table": "1d", "gather": True, "comp": True},
        # a measured, non-separable kernel
        {"name": "degrid_table2d", "kind": "degrid", "list": "pieces", "S": 24, "n": 2500000, "uneven": False,
         "ny": 384, "nx": 448, "nz": 6, "dtype": "c64", "table": "2d", "gather": False, "comp": False},
        # gridding of dense tracks (imaging)
        {"name": "grid_lines_3m", "kind": "grid", "list": "line", "S": 32, "n": 3200000, "uneven": False,
         "ny": 512, "nx": 512, "nz": 4, "table": "1d", "gather": False},
        # gridding of sparse coverage
        {"name": "grid_scatter_2m", "kind": "grid", "list": "scatter", "S": 16, "n": 2000000, "uneven": False,
         "ny": 512, "nx": 512, "nz": 4, "table": "1d", "gather": True},
        # one optimisation step on the subgrids: forward, loss, backward
        {"name": "train_step", "kind": "train", "list": "pieces", "S": 8, "n": 700001, "uneven": False,
         "ny": 328, "nx": 400, "nz": 5, "table": "1d", "gather": False},
        # making the stack from a sky image
        {"name": "predict_512", "kind": "predict", "S": 64, "N": 512, "nz": 4, "taper": True, "shifted": False},
        # a smaller image that is no power of two, windows off the centre
        {"name": "predict_384", "kind": "predict", "S": 21, "N": 384, "nz": 4, "taper": False, "shifted": True},
        # packing a stack for 16-bit storage
        {"name": "pack_f16", "kind": "pack", "S": 32, "ny": 512, "nx": 512, "nz": 4, "dtype": "f16"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_shape(rng):
    if rng.random() < 0.5:
        return 512, 512, 4
    return _log_int(rng, 64, 640), _log_int(rng, 64, 640), rng.choice([4, 4, 5, 6, 8])


def draw(rng):
    """A case of the same ranges: sizes over their logarithm, odd ones among them."""
    kind = rng.choice(["degrid", "degrid", "degrid", "grid", "train", "predict", "pack"])
    if kind == "predict":
        N = rng.choice([64, 96, 128, 180, 200, 256, 256, 320, 384, 400, 512, 512])
        most = max(1, min(64, (64 * 512 * 512) // (N * N)))
        return {"kind": kind, "S": _log_int(rng, 1, most), "N": N, "nz": rng.choice([1, 3, 4, 4, 4]),
                "taper": rng.random() < 0.5, "shifted": rng.random() < 0.5}
    ny, nx, nz = _draw_shape(rng)
    if kind == "pack":
        return {"kind": kind, "S": _log_int(rng, 1, 32), "ny": ny, "nx": nx, "nz": nz,
                "dtype": rng.choice(["f16", "bf16"])}
    lst = rng.choice(["line", "pieces", "scatter"])
    most = {"degrid": {"line": 16000000, "pieces": 14000000, "scatter": 4000000},
            "grid": {"line": 3200000, "pieces": 3200000, "scatter": 2000000},
            "train": {"line": 2000000, "pieces": 1000000, "scatter": 200000}}[kind][lst]
    n = _log_int(rng, 1000, most)
    S = max(1, min(_log_int(rng, 1, 96 if kind == "degrid" else 32), n // 500))
    gather = lst == "scatter" and nz == 4 and rng.random() < 0.8
    if lst == "scatter" and not gather:
        n = min(n, 400000)
    case = {"kind": kind, "list": lst, "S": S, "n": n, "uneven": rng.random() < 0.5,
            "ny": ny, "nx": nx, "nz": nz, "table": "1d", "gather": gather}
    if not gather and rng.random() < 0.15:
        case["table"] = "2d"
    if kind == "degrid":
        case["dtype"] = rng.choice(["c64", "c64", "f16", "bf16"])
        case["comp"] = rng.random() < 0.25
    return case


# ---- inputs ----------------------------------------------------------------

def _kaiser_bessel(x, support, beta):
    t = 2.0 * x / support
    arg = beta * np.sqrt(np.clip(1.0 - t * t, 0.0, None))
    return np.where(np.abs(x) <= support / 2, np.i0(arg) / np.i0(beta), 0.0)


def _offsets(oversample, support):
    return (np.arange(support)[None, :] - support // 2 + 1) - np.arange(oversample)[:, None] / oversample


@functools.lru_cache(maxsize=None)
def _tables(table):
    """(g_uv [O][8] or [O][O][8][8], g_w [128][4]), float64."""
    g_w = _kaiser_bessel(_offsets(W_OVERSAMPLE, W_SUPPORT), W_SUPPORT, 2.3 * W_SUPPORT)
    if table == "1d":
        return _kaiser_bessel(_offsets(UV_OVERSAMPLE, UV_SUPPORT), UV_SUPPORT, 2.3 * UV_SUPPORT), g_w
    off = _offsets(64, UV_SUPPORT)
    r = np.sqrt(off[:, None, :, None] ** 2 + off[None, :, None, :] ** 2)
    return _kaiser_bessel(r, UV_SUPPORT, 2.3 * UV_SUPPORT), g_w


def _generator(seed, stream):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed * 16 + stream)
    return g


def _gaussian(shape, seed, stream):
    x = torch.randn(tuple(shape) + (2,), generator=_generator(seed, stream), device=DEVICE, dtype=torch.float32)
    return torch.view_as_complex(x)


def _counts(case, rng):
    S, n = case["S"], case["n"]
    share = 10.0 ** rng.uniform(0.0, 3.0, S) if case["uneven"] else np.ones(S)
    c = np.floor(share / share.sum() * n).astype(np.int64)
    c[: n - int(c.sum())] += 1
    return c


def _coordinates(case, seed):
    """(uvw float64 [N][3], vis_offsets int64 [S + 1]) on the device."""
    rng = np.random.default_rng([seed, 7])
    counts = _counts(case, rng)
    offsets = np.concatenate([[0], np.cumsum(counts)])
    lo = np.array([3.5, 3.5, 1.0])
    hi = np.array([case["nx"] - 4.5, case["ny"] - 4.5, case["nz"] - 2.01])
    n = int(offsets[-1])
    offs = torch.from_numpy(offsets).to(DEVICE)
    if case["list"] == "scatter":
        r = torch.rand((n, 3), generator=_generator(seed, 2), device=DEVICE, dtype=torch.float64)
        return r * torch.from_numpy(hi - lo).to(DEVICE) + torch.from_numpy(lo).to(DEVICE), offs
    sizes, start, end, curve = [], [], [], []
    for c in counts:
        k = int(rng.integers(1, 9)) if case["list"] == "pieces" else 1
        for m in np.diff(np.linspace(0, int(c), k + 1).astype(np.int64)):
            sizes.append(int(m))
            a, b = rng.uniform(lo, hi), rng.uniform(lo, hi)
            start.append(a)
            end.append(b)
            if case["list"] == "pieces" and rng.random() < 0.5:        # a circular arc inside the box
                rmax = 0.5 * min(hi[0] - lo[0], hi[1] - lo[1])
                r = rng.uniform(min(5.0, 0.5 * rmax), rmax)
                curve.append([r, rng.uniform(lo[0] + r, hi[0] - r), rng.uniform(lo[1] + r, hi[1] - r),
                              rng.uniform(0.0, 2.0 * math.pi), rng.uniform(0.1, 2.0 * math.pi)])
            else:
                curve.append([0.0] * 5)
    size = torch.tensor(sizes, device=DEVICE)
    first = torch.cumsum(size, 0) - size
    piece = torch.repeat_interleave(torch.arange(len(sizes), device=DEVICE), size, output_size=n)
    t = (torch.arange(n, device=DEVICE) - first[piece]).double() / (size[piece] - 1).clamp(min=1)
    a = torch.from_numpy(np.array(start)).to(DEVICE)
    b = torch.from_numpy(np.array(end)).to(DEVICE)
    cv = torch.from_numpy(np.array(curve)).to(DEVICE)
    uvw = a[piece] + t[:, None] * (b - a)[piece]
    r, angle = cv[piece, 0], cv[piece, 3] + t * cv[piece, 4]
    arc = r > 0
    uvw[:, 0] = torch.where(arc, cv[piece, 1] + r * torch.cos(angle), uvw[:, 0])
    uvw[:, 1] = torch.where(arc, cv[piece, 2] + r * torch.sin(angle), uvw[:, 1])
    box = torch.from_numpy(np.stack([lo, hi])).to(DEVICE)
    return torch.minimum(torch.maximum(uvw, box[0]), box[1]).contiguous(), offs


def _pack(sub, dtype):
    """16-bit codes [S][ny][nx][nz][2] and the scale per subgrid."""
    x = torch.view_as_real(sub)
    scale = x.abs().amax(dim=(1, 2, 3, 4))
    return (x / scale[:, None, None, None, None]).to(torch.float16 if dtype == "f16" else torch.bfloat16), scale


def _stack_inputs(case, seed):
    return _gaussian((case["S"], case["ny"], case["nx"], case["nz"]), seed, 0)


def _sky(case, seed):
    """(image, taper, theta, uv_offsets, w_planes) of the producer."""
    N, S = case["N"], case["S"]
    rng = np.random.default_rng([seed, 4])
    img = 1e-4 * rng.standard_normal((N, N)) + 1e-5j * rng.standard_normal((N, N))
    at = (rng.integers(0, N, 300), rng.integers(0, N, 300))
    np.add.at(img, at, 10.0 ** rng.uniform(-3, 0, 300) * (1 + 0.01j * rng.standard_normal(300)))
    x = (np.arange(N) - N // 2) / (N / 2)
    bell = np.cos(0.45 * np.pi * x) ** 2 + 0.05
    taper = (1.0 / np.outer(bell, bell)).astype(np.float32) if case["taper"] else None
    dw = np.full(S, 100.0) if not case["shifted"] else rng.choice([60.0, 100.0], S)
    uv = rng.integers(-N, N, (S, 2)) if case["shifted"] else np.zeros((S, 2))
    w = np.stack([(np.arange(S) - S // 2) * 4.0 * dw, dw], axis=1)
    dev = lambda v: None if v is None else torch.from_numpy(np.ascontiguousarray(v)).to(DEVICE)
    return dev(img.astype(np.complex64)), dev(taper), 0.1, dev(uv.astype(np.int32)), dev(w)


# ---- prepare and run -------------------------------------------------------

def _plan(case):
    g_uv, g_w = _tables(case["table"])
    kw = {"g_uv": g_uv} if case["table"] == "1d" else {"g_uv2": g_uv}
    return dg.DegridPlan(shape=(case["ny"], case["nx"], case["nz"]), g_w=g_w, dtype=case.get("dtype", "c64"),
                         compensated=case.get("comp", False), gather=case["gather"], **kw)


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "predict":
        s["image"], s["taper"], s["theta"], s["uv"], s["w"] = _sky(case, seed)
        s["plan"] = dg.SubgridPredictor(n=case["N"], nz=case["nz"], subgrids_per_pass=32)
        return s
    if kind == "pack":
        s["sub"], s["dtype"] = _stack_inputs(case, seed), case["dtype"]
        return s
    s["uvw"], s["offs"] = _coordinates(case, seed)
    s["plan"], s["S"] = _plan(case), case["S"]
    if kind in ("grid", "train"):
        s["vis"] = _gaussian((case["n"],), seed, 1)
    if kind in ("degrid", "train"):
        s["sub"], s["scale"] = _stack_inputs(case, seed), None
        if case.get("dtype", "c64") != "c64":
            s["sub"], s["scale"] = _pack(s["sub"], case["dtype"])
    if kind == "train":
        s["sub"].requires_grad_()
    return s


def run(s):
    kind = s["kind"]
    if kind == "degrid":
        return s["plan"].degrid(s["sub"], s["uvw"], s["offs"], scale=s["scale"])
    if kind == "grid":
        return s["plan"].grid(s["vis"], s["uvw"], s["offs"], s["S"])
    if kind == "train":
        vis = dg.DegridFn.apply(s["sub"], s["uvw"], s["offs"], s["plan"])
        loss = torch.view_as_real(vis - s["vis"]).square().sum()
        grad, = torch.autograd.grad(loss, s["sub"])
        return vis.detach(), loss.detach(), grad
    if kind == "predict":
        return s["plan"].predict(s["image"], s["theta"], s["uv"], s["w"], taper=s["taper"])
    return dg.pack_subgrids(s["sub"], s["dtype"])


# ---- what a pass cannot do without -----------------------------------------

def work(case):
    """Bytes: every input that the path touches once, every output once.
    Flops: the factored sums (one multiply-add per term)."""
    kind = case["kind"]
    if kind == "predict":
        cells = case["S"] * case["N"] ** 2
        return {"bytes": 8 * cells * case["nz"] + (12 if case["taper"] else 8) * case["N"] ** 2,
                "flops": cells * case["nz"] * (10 * math.log2(case["N"]) + 6)}
    plane = case["ny"] * case["nx"] * case["nz"]
    if kind == "pack":
        return {"bytes": 12 * plane * case["S"], "flops": 2 * plane * case["S"]}
    n, S = case["n"], case["S"]
    elem = 8 if case.get("dtype", "c64") == "c64" else 4
    if case["list"] == "scatter":
        touched, per_vis = min(S * plane, 256 * n), 1024 + 288
    else:                           # tracks: a strip of the footprint's width along each
        pieces = 1 if case["list"] == "line" else 4
        touched, per_vis = min(S * plane, 256 * n, S * pieces * 16 * 4 * (case["nx"] + case["ny"]) // 2), 288
    table = 4 * (UV_OVERSAMPLE * 8 if case["table"] == "1d" else 64 * 64 * 64)
    byts = 24 * n + 8 * n + table
    if kind == "degrid":
        return {"bytes": byts + elem * touched, "flops": per_vis * n}
    if kind == "grid":
        return {"bytes": byts + 8 * S * plane, "flops": per_vis * n}
    return {"bytes": byts + 8 * n + 8 * touched + 8 * S * plane, "flops": (2 * per_vis + 6) * n}


# ---- tolerance and definition ----------------------------------------------

def tolerance(case):
    """Four times what 32-bit sums of the same terms in other orders differ by
    (measured against `exact`: 0.7e-7 to 1.6e-7 of the 2-norm, 2.4e-7 for the
    producer's two 1D transforms and phases); packing is exact by definition."""
    if case["kind"] == "pack":
        return "exact"
    if case["kind"] == "predict":
        return {"rel": 1e-6, "max": 2e-5}
    return {"rel": 8e-7, "max": 2e-5}


_CHUNK = 1 << 16


def _snap(q, oversample, support):
    p = torch.round(q * oversample).long()
    i = torch.div(p, oversample, rounding_mode="floor")
    return i - support // 2 + 1, p - i * oversample


def _terms(case, uvw, offs):
    """Yields (visibilities, subgrid of each, flat elements, weights [n][8][8][4])."""
    g_uv, g_w = (torch.from_numpy(np.ascontiguousarray(t)).to(DEVICE) for t in _tables(case["table"]))
    ny, nx, nz = case["ny"], case["nx"], case["nz"]
    b = torch.arange(8, device=DEVICE)
    c = torch.arange(4, device=DEVICE)
    cells = (b[:, None, None] * nx + b[None, :, None]) * nz + c[None, None, :]
    over = UV_OVERSAMPLE if case["table"] == "1d" else 64
    for i in range(0, uvw.shape[0], _CHUNK):
        at = torch.arange(i, min(i + _CHUNK, uvw.shape[0]), device=DEVICE)
        s = torch.searchsorted(offs, at, right=True) - 1
        (x0, fu), (y0, fv) = _snap(uvw[at, 0], over, 8), _snap(uvw[at, 1], over, 8)
        z0, fw = _snap(uvw[at, 2], W_OVERSAMPLE, 4)
        key = ((s * ny + y0) * nx + x0) * nz + z0
        g = g_uv[fv][:, :, None] * g_uv[fu][:, None, :] if case["table"] == "1d" else g_uv[fv, fu]
        yield at, s, key[:, None, None, None] + cells, g[:, :, :, None] * g_w[fw][:, None, None, :]


def _exact_degrid(case, uvw, offs, sub, scale=None):
    flat = torch.view_as_real(sub).reshape(-1, 2) if sub.is_complex() else sub.reshape(-1, 2)
    out = torch.empty(uvw.shape[0], 2, dtype=torch.float64, device=DEVICE)
    for at, s, cell, weight in _terms(case, uvw, offs):
        v = (flat[cell.reshape(len(at), -1)].double() * weight.reshape(len(at), -1, 1)).sum(1)
        out[at] = v if scale is None else v * scale[s].double()[:, None]
    return torch.view_as_complex(out)


def _exact_grid(case, uvw, offs, vis):
    shape = (case["S"], case["ny"], case["nx"], case["nz"], 2)
    out = torch.zeros(shape, dtype=torch.float64, device=DEVICE)
    y = torch.view_as_real(vis).double()
    for at, s, cell, weight in _terms(case, uvw, offs):
        out.view(-1, 2).index_add_(0, cell.reshape(-1), (weight[..., None] * y[at][:, None, None, None, :]).reshape(-1, 2))
    return torch.view_as_complex(out)


def _exact_predict(case, image, taper, theta, uv, w):
    N, nz = case["N"], case["nz"]
    k = torch.arange(N, device=DEVICE, dtype=torch.float64) - N // 2
    r2 = ((k * theta / N) ** 2)[None, :] + ((k * theta / N) ** 2)[:, None]
    nm1 = torch.where(r2 < 1.0, -r2 / (1.0 + torch.sqrt((1.0 - r2).clamp(min=0.0))), 0.0)
    sky = image.to(torch.complex128) * (r2 < 1.0)
    if taper is not None:
        sky = sky * taper.double()
    out = torch.empty((case["S"], N, N, nz), dtype=torch.complex128, device=DEVICE)
    for s in range(case["S"]):
        u0, v0 = (int(v) for v in uv[s].cpu())
        for c in range(nz):
            turns = -(w[s, 0] + c * w[s, 1]) * nm1
            plane = sky * torch.polar(torch.ones_like(turns), 2.0 * math.pi * (turns - torch.round(turns)))
            grid = torch.fft.fftshift(torch.fft.fft2(torch.fft.ifftshift(plane)))
            out[s, :, :, c] = torch.roll(grid, (-v0, -u0), (0, 1))
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "predict":
        return _exact_predict(case, *_sky(case, seed))
    if kind == "pack":
        x = torch.view_as_real(_stack_inputs(case, seed)).double()
        scale = x.abs().amax(dim=(1, 2, 3, 4))
        return x / scale[:, None, None, None, None], scale
    uvw, offs = _coordinates(case, seed)
    if kind == "grid":
        return _exact_grid(case, uvw, offs, _gaussian((case["n"],), seed, 1))
    sub, scale = _stack_inputs(case, seed), None
    if kind == "degrid" and case["dtype"] != "c64":
        sub, scale = _pack(sub, case["dtype"])
    vis = _exact_degrid(case, uvw, offs, sub, scale)
    if kind == "degrid":
        return vis
    diff = vis - _gaussian((case["n"],), seed, 1)
    return vis, torch.view_as_real(diff).square().sum(), 2.0 * _exact_grid(case, uvw, offs, diff)
