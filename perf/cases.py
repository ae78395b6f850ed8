"""Performance cases: the calls a user of this framework makes, over the range of sizes, types and modes it serves.

A case is a dict of plain values whose "kind" selects the call:
  frame      one whole frame of an in-situ renderer: sampling bricks of the time step's volume, K compact
             sub-VDIs, their composite and its flattened image (the generating view);
  generate   sub-VDI generation alone from resident bricks, with a fixed gamma, the per-ray search, the learned
             choice, or the search under a non-convex ownership map (all PEs sample one whole-volume brick);
  gen_batch  many uneven generation requests in one batched call;
  composite  K depth-sorted lists per pixel, from any source and overlapping in depth, composited and flattened;
  comp_batch many uneven compositing requests in one batched call, each flattened;
  render     a generated VDI rendered from another viewpoint;
  train      one training step of the learned-gamma model from a checkpoint.
"""
import math
import os
import struct

import torch

import paper_2206_14503_gb300 as vdi

DEV = "cuda"
CKPT = os.path.join(os.path.dirname(os.path.abspath(vdi.__file__)), "models", "gamma_ns32_k16.ckpt")
STEP, REF_LEN, FOVY = 0.5, 1.0, 45.0
PARAMS, WEIGHTS, MOMENT1, MOMENT2, STEPS = 6849, 0, 41472, 69120, 96768  # a model buffer's parts (bytes)
REC = {0: 24, 1: 16}  # bytes of an FP32 / FP16 record
SEARCH, FIXED = "search", "fixed"


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest useful frame (a preview): launches and latency count
        dict(name="frame_64", kind="frame", dims="64x64x64", u16=False, grid="1x1x2", w=128, h=128, n_s=8, prec=0,
             mode=FIXED, gamma=0.02),
        # the benchmark's frame
        dict(name="frame_512", kind="frame", dims="512x512x512", u16=True, grid="2x2x2", w=1920, h=1080, n_s=20,
             prec=0, mode=SEARCH, gamma=0.0),
        # odd sizes in every direction, float volume, FP16 records
        dict(name="frame_ragged_f16", kind="frame", dims="201x157x251", u16=False, grid="1x2x3", w=853, h=479,
             n_s=12, prec=1, mode=SEARCH, gamma=0.0),
        # one process, interactive gamma slider: one march and the emission
        dict(name="generate_fixed_384", kind="generate", dims="384x384x384", u16=True, grid="1x1x1", w=1280, h=720,
             n_s=25, prec=0, mode=FIXED, gamma=0.05),
        # the learned-gamma workload: the largest volume, gamma predicted per tile and refined per ray
        dict(name="generate_learned_1024", kind="generate", dims="1024x1024x1024", u16=True, grid="4x2x2", w=1920,
             h=1080, n_s=32, prec=0, mode="learned", gamma=0.0),
        # a simulation whose domains are not boxes: blocks of 32 cells dealt out to four PEs
        dict(name="generate_owned_256", kind="generate", dims="256x256x256", u16=True, grid="2x2x1", w=1024, h=768,
             n_s=16, prec=0, mode="owned", gamma=0.0),
        # a server's requests: volumes, decompositions and images of several sizes at once
        dict(name="generate_batch_6", kind="gen_batch", n=6, side_lo=128, side_hi=256, w_lo=256, w_hi=1280, prec=0),
        # dense overlapping lists of 32 PEs: the longest lists a pixel's stage holds
        dict(name="composite_dense_k32", kind="composite", w=640, h=480, k=32, n_s=32, prec=0, dense=True),
        # ragged list lengths, odd image, FP16 storage
        dict(name="composite_k12_f16", kind="composite", w=801, h=601, k=12, n_s=24, prec=1, dense=False),
        # a server's compositing requests of several K, N_S and image sizes at once
        dict(name="composite_batch_5", kind="comp_batch", n=5, w_lo=192, w_hi=640, k_lo=2, k_hi=32, prec=0),
        # looking around a streamed VDI between two of its updates
        dict(name="render_20deg", kind="render", dims="256x256x256", grid="1x2x2", w=1920, h=1080, n_s=20, prec=0,
             degrees=20.0),
        # the learned-gamma model's training step at its mini-batch size
        dict(name="train_65536", kind="train", rows=65536),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _text(sizes):
    return "x".join(str(n) for n in sizes)


def _plain(case):
    """The case with its sizes ("64x64x64") as lists."""
    return {k: [int(n) for n in v.split("x")] if k in ("dims", "grid") else v for k, v in case.items()}


def _grid(rng, most=16):
    while True:
        g = [rng.choice((1, 2, 3, 4)), rng.choice((1, 2)), rng.choice((1, 2, 3))]
        if g[0] * g[1] * g[2] <= most:
            return _text(g)


def draw(rng):
    kind = rng.choice(("frame", "frame", "generate", "generate", "gen_batch", "composite", "composite", "comp_batch",
                       "render", "train"))
    prec = rng.choice((0, 0, 1))
    if kind in ("frame", "generate"):
        side = _log(rng, 48, 448)
        dims = _text(max(24, int(side * rng.uniform(0.6, 1.15))) for _ in range(3))
        w = _log(rng, 96, 1900)
        c = dict(kind=kind, dims=dims, u16=rng.random() < 0.6, grid=_grid(rng), w=w,
                 h=max(64, int(w * rng.uniform(0.4, 0.8))), n_s=rng.randint(4, 40), prec=prec,
                 mode=rng.choice((SEARCH, SEARCH, FIXED) if kind == "frame" else (SEARCH, FIXED, "learned", "owned")),
                 gamma=round(rng.uniform(0.005, 0.15), 4))
        return c
    if kind == "gen_batch":
        lo = _log(rng, 48, 160)
        w = _log(rng, 128, 500)
        return dict(kind=kind, n=rng.randint(2, 6), side_lo=lo, side_hi=lo + rng.randint(16, 96), w_lo=w,
                    w_hi=w + rng.randint(50, 700), prec=prec)
    if kind == "composite":
        k, n_s, dense = rng.randint(1, 48), rng.randint(4, 32), rng.random() < 0.3
        w = _log(rng, 64, 1200)
        h = max(33, int(w * rng.uniform(0.4, 0.9)))
        while w * h * k * n_s > 200_000_000:
            w, h = int(w * 0.8), int(h * 0.8)
        return dict(kind=kind, w=w, h=h, k=k, n_s=n_s, prec=prec, dense=dense)
    if kind == "comp_batch":
        w = _log(rng, 96, 320)
        return dict(kind=kind, n=rng.randint(2, 5), w_lo=w, w_hi=w + rng.randint(20, 240), k_lo=2,
                    k_hi=rng.randint(4, 32), prec=prec)
    if kind == "render":
        side = _log(rng, 64, 256)
        w = _log(rng, 160, 1900)
        return dict(kind=kind, dims=_text((side, side + rng.randint(0, 40), side - rng.randint(0, 30))), grid=_grid(rng, 8),
                    w=w, h=max(90, int(w * rng.uniform(0.45, 0.75))), n_s=rng.randint(6, 32), prec=prec,
                    degrees=round(rng.uniform(2.0, 50.0), 2))
    return dict(kind="train", rows=_log(rng, 2000, 65536) | 1)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _gen(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1009 + salt)
    return g


def _volume(dims, u16, seed, salt=0):
    """Gaussian blobs and three octaves of smooth noise, normalised to [0, 1] (a simulation's scalar field); float32,
    or the bit pattern of round(65535 v) as int16."""
    X, Y, Z = dims
    g = _gen(seed, 1 + salt)
    blobs = 16 if max(dims) < 96 else (64 if max(dims) < 700 else 128)
    cen = torch.rand((blobs, 3), generator=g, device=DEV)
    sig = 0.03 + 0.12 * torch.rand((blobs, 3), generator=g, device=DEV)

    def axis(n, a):
        u = torch.arange(n, dtype=torch.float32, device=DEV) / (n - 1)
        return torch.exp(-(u[None, :] - cen[:, a:a + 1]) ** 2 / (2 * sig[:, a:a + 1] ** 2))

    gx, gy, gz = axis(X, 0), axis(Y, 1), axis(Z, 2)
    v = ((gz[:, :, None] * gy[:, None, :]).reshape(blobs, Z * Y).t() @ gx).view(Z, Y, X)
    for o in range(3 if max(dims) < 700 else 4):
        f = 4 << o
        lat = torch.rand((1, 1, f + 1, f + 1, f + 1), generator=g, device=DEV)
        v += 0.1 * 0.5 ** o * torch.nn.functional.interpolate(lat, size=(Z, Y, X), mode="trilinear",
                                                              align_corners=True)[0, 0]
    lo, hi = v.min(), v.max()
    v = (v - lo) / (hi - lo)
    if not u16:
        return v.contiguous()
    u = torch.floor(v * 65535.0 + 0.5).clamp_(0, 65535).to(torch.int32)
    return (u - 65536 * (u > 32767).int()).to(torch.int16).contiguous()


def _table():
    """The transfer function a user has set: five opacity bumps over a hue ramp, nothing below v = 0.2."""
    v = torch.arange(256, dtype=torch.float64) / 255.0
    al = torch.zeros_like(v)
    for m, s, a in ((0.31, 0.04, 0.30), (0.44, 0.03, 0.45), (0.58, 0.05, 0.25), (0.72, 0.035, 0.55),
                    (0.90, 0.06, 0.35)):
        al += a * torch.exp(-(v - m) ** 2 / (2 * s * s))
    al = torch.where((v >= 0.2) & (al >= 1e-3), al.clamp(max=0.6), torch.zeros_like(al))
    hue = (200.0 + 300.0 * v) / 60.0
    ch = [((hue + s) % 6.0 - 3.0).abs() - 1.0 for s in (0.0, 4.0, 2.0)]
    rgb = [0.2 + 0.8 * c.clamp(0.0, 1.0) for c in ch]
    return torch.stack(rgb + [al], dim=-1).to(torch.float32).contiguous()


class _Cam:
    def __init__(self, eye, center, width, height):
        self.eye, self.center, self.up = tuple(eye), tuple(center), (0.0, 0.0, 1.0)
        self.fovy_deg, self.width, self.height = FOVY, width, height


def _orbit(dims, w, h, seed, salt=0, turn=0.0):
    """A view of the volume's orbit (1.8 half-diagonals from its centre), turned by `turn` degrees about it."""
    a, b = torch.rand(2, generator=torch.Generator().manual_seed(int(seed) * 7919 + salt), dtype=torch.float64).tolist()
    az, el = 2 * math.pi * a + math.radians(turn), (math.pi / 6) * (2 * b - 1)
    c = [0.5 * (d - 1) for d in dims]
    r = 0.9 * math.sqrt(sum((d - 1) ** 2 for d in dims))
    return _Cam((c[0] + r * math.cos(el) * math.cos(az), c[1] + r * math.cos(el) * math.sin(az), c[2] + r * math.sin(el)),
                c, w, h)


def _lists(npix, k, n_s, prec, dense, seed):
    """K sub-VDIs of depth-sorted, non-overlapping records on unit depth (those of different PEs overlap)."""
    out = []
    for e in range(k):
        g = _gen(seed, 100 + e)
        cnt = (torch.full((npix,), n_s, dtype=torch.int32, device=DEV) if dense
               else torch.randint(0, n_s + 1, (npix,), generator=g, device=DEV, dtype=torch.int32))
        off = torch.zeros(npix + 1, dtype=torch.int64, device=DEV)
        off[1:] = torch.cumsum(cnt.to(torch.int64), 0)
        fbs, cols = [], []
        for p0 in range(0, npix, 1 << 18):
            n = min(npix - p0, 1 << 18)
            t = torch.rand((n, 2 * n_s), generator=g, device=DEV)
            live = torch.arange(2 * n_s, device=DEV)[None, :] < 2 * cnt[p0:p0 + n, None]
            t = torch.where(live, t, torch.full_like(t, 2.0)).sort(dim=1)[0].view(n, n_s, 2)
            a = torch.rand((n, n_s, 1), generator=g, device=DEV)
            c = torch.cat([a * torch.rand((n, n_s, 3), generator=g, device=DEV), a], dim=-1)
            keep = live.view(n, n_s, 2)[..., 0]
            fbs.append(t[keep])
            cols.append(c[keep])
        fb, col = torch.cat(fbs).contiguous(), torch.cat(cols).contiguous()
        if prec == 1:
            half = torch.cat([col[:, :3], -torch.log2(1.0 - col[:, 3:])], dim=-1).to(torch.float16)
            col = torch.cat([fb.view(torch.int32), half.view(torch.int32)], dim=-1).contiguous()
            fb = None
        out.append(vdi.Compact.from_tensors(cnt, off, col, fb, prec))
    return out


# ---------------------------------------------------------------------------
# States: what a program holds before the call
# ---------------------------------------------------------------------------
def _boxes(case):
    return vdi.vdi_split_boxes(case["dims"], case["grid"])


def _bricks(case, vol):
    if case.get("mode") == "owned":  # every PE samples the whole volume's brick
        b = vdi.vdi_split_boxes(case["dims"], [1, 1, 1])
        one = vdi.Bricks(vol, case["dims"], b)
        return one, [one.bricks[0]] * _pes(case)
    br = vdi.Bricks(vol, case["dims"], _boxes(case))
    return br, list(br.bricks)


def _pes(case):
    return case["grid"][0] * case["grid"][1] * case["grid"][2]


def _sub_vdis(parts, prec):
    """Buffers of the sub-VDIs of several requests (k PEs, pixels, records a PE's sub-VDI may hold), each kind of buffer
    in one allocation: (the allocations, per request its PEs' sub-VDIs)."""
    pes = sum(k for k, _, _ in parts)
    npix, recs = sum(k * n for k, n, _ in parts), sum(k * c for k, _, c in parts)
    out = {"counts": torch.zeros(npix, dtype=torch.int32, device=DEV),
           "offsets": torch.zeros(npix + pes, dtype=torch.int64, device=DEV),
           "gamma": torch.zeros(npix, dtype=torch.float32, device=DEV),
           "rgba": torch.zeros((recs, 4), dtype=torch.int32 if prec else torch.float32, device=DEV)}
    if not prec:
        out["fb"] = torch.zeros((recs, 2), dtype=torch.float32, device=DEV)
    got, p, o, r = [], 0, 0, 0
    for k, n, c in parts:
        got.append([])
        for _ in range(k):
            got[-1].append(vdi.Compact.from_tensors(out["counts"][p:p + n], out["offsets"][o:o + n + 1],
                                                    out["rgba"][r:r + c], None if prec else out["fb"][r:r + c], prec,
                                                    out["gamma"][p:p + n]))
            p, o, r = p + n, o + n + 1, r + c
    return out, got


def _gamma(case):
    return case["gamma"] if case["mode"] == FIXED else vdi.VDI_GAMMA_SEARCH


def prepare(case, seed):
    return _prepare(_plain(case), seed)


def _prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "params": vdi.make_params(step=STEP, ref_len=REF_LEN)}
    if kind in ("frame", "generate", "render"):
        w, h, n_s, prec = case["w"], case["h"], case["n_s"], case["prec"]
        full = dict({"u16": True, "mode": SEARCH, "gamma": 0.0}, **case)
        k, npix = _pes(case), w * h
        s["lut"] = _table().to(DEV)
        vol = _volume(case["dims"], full["u16"], seed)
        s["bricks"], s["list"] = _bricks(full, vol)
        s["arr"] = (vdi.vdi_brick * k)(*s["list"])
        cam = _orbit(case["dims"], w, h, seed)
        s["cam"] = vdi.make_camera(cam)
        # a PE's box covers a part of the image: room for that
        s["out"], s["outs"] = _sub_vdis([(k, npix, math.ceil(npix * n_s * min(1.0, 2.0 / math.sqrt(k))))], prec)
        s["structs"] = [o.struct() for o in s["outs"][0]]
        size = vdi.vdi_learned_workspace if full["mode"] == "learned" else vdi.vdi_generate_workspace
        s["ws"] = vdi.Workspace(size(k, w, h))
        if kind == "frame":
            s["vol"] = vol
        if kind in ("frame", "render"):
            s["reg"] = vdi.Regular(npix, n_s, prec)
            s["wsc"] = vdi.Workspace(vdi.vdi_composite_workspace(k, w, h, n_s))
            s["img"] = torch.zeros((npix, 4), dtype=torch.float32, device=DEV)
        if full["mode"] == "learned":
            s["model"] = torch.zeros(vdi.vdi_model_bytes(), dtype=torch.uint8, device=DEV)
            vdi.check(vdi.vdi_model_load(s["model"].data_ptr(), CKPT), "model")
        if full["mode"] == "owned":
            block = max(8, 1 << (max(case["dims"]) // 8).bit_length() - 1)
            nb = [-(-(d - 1) // block) for d in case["dims"]]
            z, y, x = torch.meshgrid(*(torch.arange(n, device=DEV) for n in nb[::-1]), indexing="ij")
            s["owner"] = ((x + y + z) % k).to(torch.uint8).contiguous()
            s["own"] = vdi.vdi_ownership(s["owner"].data_ptr(), block, tuple(nb))
        if kind == "render":  # the VDI a viewer holds: generated once, before the looking around
            _generate(s, full)
            _composite(s, full)
            del s["bricks"], s["list"], s["arr"], s["out"], s["outs"], s["structs"], s["ws"], s["wsc"]
            s["view"] = vdi.make_camera(_orbit(case["dims"], w, h, seed, turn=case["degrees"]))
    elif kind == "gen_batch":
        reqs = _gen_requests(case)
        s["lut"], s["keep"], items = _table().to(DEV), [], []
        s["out"], parts = _sub_vdis([(math.prod(q["grid"]), q["w"] * q["h"], q["w"] * q["h"] * q["n_s"]) for q in reqs],
                                    case["prec"])
        for r, q in enumerate(reqs):
            br = vdi.Bricks(_volume(q["dims"], True, seed, 10 * r), q["dims"], vdi.vdi_split_boxes(q["dims"], q["grid"]))
            s["keep"].append(br)
            items.append((br.bricks, s["lut"].data_ptr(), vdi.make_camera(_orbit(q["dims"], q["w"], q["h"], seed, r)),
                          q["n_s"], vdi.VDI_GAMMA_SEARCH, [o.struct() for o in parts[r]]))
        s["reqs"] = vdi.GenRequests(items)
        s["host"] = vdi.vdi_gen_batch_table_pack(s["reqs"], s["params"])
        s["dev"] = torch.frombuffer(bytearray(s["host"]), dtype=torch.uint8).to(DEV)
        s["ws"] = vdi.Workspace(vdi.vdi_generate_batched_workspace(s["host"]))
    elif kind == "composite":
        npix = case["w"] * case["h"]
        s["outs"] = _lists(npix, case["k"], case["n_s"], case["prec"], case["dense"], seed)
        s["structs"] = [o.struct() for o in s["outs"]]
        s["reg"] = vdi.Regular(npix, case["n_s"], case["prec"])
        s["wsc"] = vdi.Workspace(vdi.vdi_composite_workspace(case["k"], case["w"], case["h"], case["n_s"]))
        s["img"] = torch.zeros((npix, 4), dtype=torch.float32, device=DEV)
    elif kind == "comp_batch":
        s["keep"], items = [], []
        for r, q in enumerate(_comp_requests(case)):
            npix = q["w"] * q["h"]
            ins = _lists(npix, q["k"], q["n_s"], case["prec"], False, seed * 31 + r)
            reg = vdi.Regular(npix, q["n_s"], case["prec"])
            img = torch.zeros((npix, 4), dtype=torch.float32, device=DEV)
            s["keep"].append((q, ins, reg, img))
            items.append(([i.struct() for i in ins], q["w"], q["h"], reg.struct(), 0))
        s["reqs"] = vdi.Requests(items)
        s["host"] = vdi.vdi_batch_table_pack(s["reqs"])
        s["dev"] = torch.frombuffer(bytearray(s["host"]), dtype=torch.uint8).to(DEV)
        s["ws"] = vdi.Workspace(vdi.vdi_composite_batched_workspace(s["host"]))
    else:
        s["model"] = torch.zeros(vdi.vdi_model_bytes(), dtype=torch.uint8, device=DEV)
        vdi.check(vdi.vdi_model_load(s["model"].data_ptr(), CKPT), "model")
        s["x"], s["y"], s["valid"] = _rows(case["rows"], seed)
        s["loss"] = torch.zeros(1, dtype=torch.float32, device=DEV)
        s["ws"] = vdi.Workspace(vdi.vdi_mlp_train_workspace(case["rows"]))
    return s


def _gen_requests(case):
    """Uneven requests between the case's bounds, the same for every seed (the service's clients)."""
    grids, out = ([1, 1, 1], [1, 1, 2], [1, 2, 2], [2, 2, 2], [4, 2, 2]), []
    for r in range(case["n"]):
        f, g = (r * 0.618034) % 1.0, (r * 0.414214 + 0.3) % 1.0
        side = int(case["side_lo"] + f * (case["side_hi"] - case["side_lo"]))
        w = int(case["w_lo"] + g * (case["w_hi"] - case["w_lo"]))
        out.append(dict(dims=[side, side + r, max(24, side - 3 * r)], grid=grids[r % 5], w=w, h=int(w * (0.5 + 0.3 * f)),
                        n_s=8 + int(32 * g)))
    return out


def _comp_requests(case):
    out = []
    for r in range(case["n"]):
        f, g = (r * 0.618034) % 1.0, (r * 0.414214 + 0.3) % 1.0
        w = int(case["w_lo"] + g * (case["w_hi"] - case["w_lo"]))
        k = case["k_hi"] if r == 0 else int(case["k_lo"] + f * (case["k_hi"] - case["k_lo"]))
        out.append(dict(w=w, h=int(w * (0.5 + 0.3 * f)), k=k, n_s=8 + int(24 * g)))
    return out


def _rows(n, seed):
    """Tile features as the feature kernel gives them (a sparse histogram, depths, counts) and labels near a smooth
    function of them; one row in twenty is a tile without samples."""
    g = _gen(seed, 3)
    x = torch.rand((n, 40), generator=g, device=DEV)
    hist = x[:, :32] ** 6
    x[:, :32] = hist / hist.sum(dim=1, keepdim=True)
    x[:, 37] = 0.5
    y = -4.0 - 3.0 * x[:, 36] + 2.0 * x[:, 39] + 0.5 * torch.randn(n, generator=g, device=DEV)
    return x.contiguous(), y.contiguous(), (torch.rand(n, generator=g, device=DEV) > 0.05).to(torch.uint8)


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def _part(model, at):
    return model[at:at + 4 * PARAMS].view(torch.float32)


def _offset():
    return 0.0  # the shipped model's calibrated offset


def _generate(s, case):
    a = (s["arr"], s["lut"].data_ptr(), s["cam"], case["n_s"])
    st = s["ws"]
    stream = torch.cuda.current_stream()
    if case["mode"] == "learned":
        vdi.check(vdi.vdi_choose_gamma_learned(*a, s["model"].data_ptr(), _offset(), s["structs"], s["params"], st.ptr,
                                               st.nbytes, stream), "learned")
        own = vdi.vdi_learned_workspace(_pes(case), case["w"], case["h"]) - vdi.vdi_generate_workspace(
            _pes(case), case["w"], case["h"])  # the generation's part of the workspace, with its recorded spans
        vdi.check(vdi.vdi_generate(*a, vdi.VDI_GAMMA_CHOSEN, s["structs"], s["params"], st.ptr + own, st.nbytes - own,
                                   stream), "generate")
    elif case["mode"] == "owned":
        vdi.check(vdi.vdi_generate_owned(*a, _gamma(case), s["own"], s["structs"], s["params"], st.ptr, st.nbytes,
                                         stream), "generate")
    else:
        vdi.check(vdi.vdi_generate(*a, _gamma(case), s["structs"], s["params"], st.ptr, st.nbytes, stream), "generate")


def _composite(s, case):
    stream = torch.cuda.current_stream()
    vdi.check(vdi.vdi_composite(s["structs"], case["w"], case["h"], s["reg"].struct(), s["params"], s["wsc"].ptr,
                                s["wsc"].nbytes, stream), "composite")


def _flatten(reg, w, h, img):
    vdi.check(vdi.vdi_render_view(reg.struct(), w, h, vdi.vdi_camera(), None, img.data_ptr(),
                                  torch.cuda.current_stream()), "flatten")


def _records(o):
    return {k: v for k, v in (("counts", o.counts), ("gamma", o.gamma), ("rgba", o.rgba), ("fb", o.fb)) if v is not None}


def run(state):
    s, case = state, state["case"]
    kind = case["kind"]
    stream = torch.cuda.current_stream()
    if kind == "frame":
        s["bricks"].rebuild(s["vol"], stream)
        _generate(s, case)
        _composite(s, case)
        _flatten(s["reg"], case["w"], case["h"], s["img"])
        return dict(_records(s["reg"]), image=s["img"])
    if kind == "generate":
        _generate(s, case)
        return s["out"]
    if kind == "gen_batch":
        vdi.check(vdi.vdi_generate_batched(s["dev"].data_ptr(), s["host"], s["ws"].ptr, s["ws"].nbytes, stream), "batch")
        return s["out"]
    if kind == "composite":
        _composite(s, case)
        _flatten(s["reg"], case["w"], case["h"], s["img"])
        return dict(_records(s["reg"]), image=s["img"])
    if kind == "comp_batch":
        vdi.check(vdi.vdi_composite_batched(s["dev"].data_ptr(), s["host"], s["params"], s["ws"].ptr, s["ws"].nbytes,
                                            stream), "batch")
        for q, _, reg, img in s["keep"]:
            _flatten(reg, q["w"], q["h"], img)
        return [dict(_records(reg), image=img) for _, _, reg, img in s["keep"]]
    if kind == "render":
        vdi.check(vdi.vdi_render_view(s["reg"].struct(), case["w"], case["h"], s["cam"], s["view"], s["img"].data_ptr(),
                                      stream), "render")
        return {"image": s["img"]}
    vdi.check(vdi.vdi_mlp_train_step(s["model"].data_ptr(), s["x"].data_ptr(), s["y"].data_ptr(), s["valid"].data_ptr(),
                                     case["rows"], 3e-4, s["loss"].data_ptr(), s["ws"].ptr, s["ws"].nbytes, stream),
              "train")
    return {"weights": _part(s["model"], WEIGHTS), "moment1": _part(s["model"], MOMENT1),
            "moment2": _part(s["model"], MOMENT2), "loss": s["loss"]}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def _gen_work(dims, w, h, k, n_s, prec):
    """Reads one value per node, marches the rays' samples once (28 operations each, a state-machine step of 24 for the
    half of them that is not transparent) and writes counts, gamma, offsets and about n_s / 2 records where a ray meets
    a PE's box.  The mean chord and the projected area of a box are its volume over a quarter of its surface and that."""
    X, Y, Z = dims
    area, vol = 0.5 * (X * Y + Y * Z + X * Z), float(X * Y * Z)
    dist = 0.9 * math.sqrt(X * X + Y * Y + Z * Z)
    screen = (2 * dist * math.tan(math.radians(FOVY / 2))) ** 2 * w / h
    hit = min(1.0, area / screen) * w * h
    samples = hit * vol / area / STEP
    lists = hit * k ** (1.0 / 3.0)
    return 4 * vol + w * h * k * 16 + lists * 0.5 * n_s * REC[prec], samples * (28 + 0.5 * 24)


def _comp_work(npix, k, n_s, prec, mean):
    recs = npix * k * mean
    return npix * k * 12 + recs * REC[prec] + npix * (n_s * REC[prec] + 8 + 16), recs * 24


def work(case):
    case = _plain(case)
    kind = case["kind"]
    if kind in ("frame", "generate"):
        b, f = _gen_work(case["dims"], case["w"], case["h"], _pes(case), case["n_s"], case["prec"])
        if kind == "frame":
            npix = case["w"] * case["h"]
            b += npix * (case["n_s"] * REC[case["prec"]] + 8 + 16) - (2 if case["u16"] else 0) * math.prod(case["dims"])
    elif kind == "gen_batch":
        parts = [_gen_work(q["dims"], q["w"], q["h"], math.prod(q["grid"]), q["n_s"], case["prec"])
                 for q in _gen_requests(case)]
        b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
    elif kind == "composite":
        b, f = _comp_work(case["w"] * case["h"], case["k"], case["n_s"], case["prec"],
                          case["n_s"] * (1.0 if case["dense"] else 0.5))
    elif kind == "comp_batch":
        parts = [_comp_work(q["w"] * q["h"], q["k"], q["n_s"], case["prec"], 0.5 * q["n_s"]) for q in _comp_requests(case)]
        b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
    elif kind == "render":
        npix = case["w"] * case["h"]
        # half of the pixels hold a list; a ray crosses about sin(turn) of the image's columns
        b = npix * (4 + 0.5 * 0.5 * case["n_s"] * REC[case["prec"]] + 16)
        f = npix * 0.5 * max(2.0, case["w"] * math.sin(math.radians(case["degrees"])) * 0.5) * 30
    else:
        b, f = case["rows"] * (40 * 4 + 5) + PARAMS * 4 * 6, case["rows"] * 6 * 6784
    return {"bytes": float(b), "flops": float(f)}


# ---------------------------------------------------------------------------
# The same in 64 bits, in plain torch.  A list's records are decided by comparisons against a searched threshold, so a
# rounding may give another (equally valid) list: they have no value in 64 bits.  Their flattened image has one whatever
# the list: "over" is associative, so it is the volume rendering of the samples (the composite of the pieces).
# ---------------------------------------------------------------------------
def _basis(cam):
    def unit(v):
        n = math.sqrt(sum(x * x for x in v))
        return [x / n for x in v]

    def cross(a, b):
        return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]

    f = unit([c - e for c, e in zip(cam.center, cam.eye)])
    r = unit(cross(f, cam.up))
    return f, r, cross(r, f)


def _rays(cam):
    """Unit directions [3][h * w] of the pixels' centre rays, in 64 bits."""
    f, r, u = _basis(cam)
    th = math.tan(math.radians(cam.fovy_deg) / 2)
    i = torch.arange(cam.width, dtype=torch.float64, device=DEV)
    j = torch.arange(cam.height, dtype=torch.float64, device=DEV)
    x = (((2 * i + 1) / cam.width - 1) * th * cam.width / cam.height)[None, :].expand(cam.height, -1).reshape(-1)
    y = ((1 - (2 * j + 1) / cam.height) * th)[:, None].expand(-1, cam.width).reshape(-1)
    d = [f[a] + x * r[a] + y * u[a] for a in range(3)]
    n = torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
    return [c / n for c in d]


def _dvr(case, seed):
    """Direct volume rendering of the frame's samples."""
    X, Y, Z = case["dims"]
    vol = _volume(case["dims"], case["u16"], seed).reshape(-1)
    lut = _table().to(DEV).double()
    lut[:, 3] = 1 - (1 - lut[:, 3]) ** (STEP / REF_LEN)
    cam = _orbit(case["dims"], case["w"], case["h"], seed)
    d = _rays(cam)
    tin, tout = torch.zeros_like(d[0]), torch.full_like(d[0], 1e30)
    for a, n in enumerate((X, Y, Z)):
        t0, t1 = -cam.eye[a] / d[a], (n - 1 - cam.eye[a]) / d[a]
        tin, tout = torch.maximum(tin, torch.minimum(t0, t1)), torch.minimum(tout, torch.maximum(t0, t1))
    live = (tin < tout).nonzero()[:, 0]
    d, tin, tout = [c[live] for c in d], tin[live], tout[live]
    img = torch.zeros((case["w"] * case["h"], 4), dtype=torch.float64, device=DEV)
    col, alpha = torch.zeros((live.numel(), 3), dtype=torch.float64, device=DEV), torch.zeros_like(tin)
    for k in range(int(torch.ceil((tout - tin).max() / STEP)) + 1 if live.numel() else 0):
        t = tin + (k + 0.5) * STEP
        on = (t < tout).nonzero()[:, 0]
        if not on.numel():
            break
        c, w = [], []
        for a, n in enumerate((X, Y, Z)):
            p = cam.eye[a] + t[on] * d[a][on]
            i = p.floor().clamp(0, n - 2)
            c.append(i.long())
            w.append((p - i).clamp(0.0, 1.0))
        v = 0.0
        for dz in (0, 1):
            for dy in (0, 1):
                for dx in (0, 1):
                    q = vol[((c[2] + dz) * Y + c[1] + dy) * X + c[0] + dx].double()
                    if case["u16"]:
                        q = torch.where(q < 0, q + 65536.0, q) / 65535.0
                    v = v + q * (w[0] if dx else 1 - w[0]) * (w[1] if dy else 1 - w[1]) * (w[2] if dz else 1 - w[2])
        x = (v * 255.0).clamp(0.0, 255.0)
        i = x.floor().clamp(max=254).long()
        e = lut[i] + (x - i)[:, None] * (lut[i + 1] - lut[i])
        T = (1 - alpha[on])[:, None]
        col[on] += T * e[:, :3] * e[:, 3:]
        alpha[on] += T[:, 0] * e[:, 3]
    img[live] = torch.cat([col, alpha[:, None]], dim=-1)
    return img.cpu().numpy()


def _flat_lists(ins, npix, n_s, prec):
    """The K lists of every pixel cut at all bounds, mixed where they overlap, and composited front to back."""
    img = torch.zeros((npix, 4), dtype=torch.float64, device=DEV)
    step = max(1, int(4e7 / (2 * len(ins) * n_s)))
    for p0 in range(0, npix, step):
        p1 = min(npix, p0 + step)
        t, dm = [], []
        for o in ins:
            i = torch.arange(n_s, device=DEV)[None, :]
            live = i < o.counts[p0:p1, None]
            r = torch.where(live, o.offsets[p0:p1, None] + i, torch.zeros_like(i))
            if prec == 1:
                raw = o.rgba[r]
                fb = raw[..., :2].contiguous().view(torch.float32).double()
                c = raw[..., 2:].contiguous().view(torch.float16).double()
                tau, rgb = c[..., 3], c[..., :3]
                A = -torch.expm1(-tau * math.log(2.0))
            else:
                fb, c = o.fb[r].double(), o.rgba[r].double()
                A, rgb = c[..., 3], c[..., :3]
                tau = -torch.log2(1 - A)
            ok = live & (fb[..., 1] > fb[..., 0]) & (A > 0)
            mu = torch.where(ok, tau / (fb[..., 1] - fb[..., 0]), torch.zeros_like(tau))
            m = torch.stack([mu] + [torch.where(ok, mu * rgb[..., q] / A, torch.zeros_like(mu)) for q in range(3)], -1)
            fb = torch.where(ok[..., None], fb, torch.full_like(fb, 2.0))
            t += [fb[..., 0], fb[..., 1]]
            dm += [m, -m]
        t, order = torch.cat(t, dim=1).sort(dim=1)
        dm = torch.cat(dm, dim=1).gather(1, order[..., None].expand(-1, -1, 4)).cumsum(dim=1)[:, :-1]
        dt = t[:, 1:] - t[:, :-1]
        M = dm[..., 0].clamp(min=0.0)
        w = torch.where(M > 1e-9, -torch.expm1(-M * dt * math.log(2.0)) / M.clamp(min=1e-9), dt * math.log(2.0))
        L = (M * dt).cumsum(dim=1)
        T = torch.exp2(-(L - M * dt))
        img[p0:p1, :3] = (T * w).unsqueeze(-1).mul(dm[..., 1:]).sum(dim=1)
        img[p0:p1, 3] = -torch.expm1(-L[:, -1] * math.log(2.0))
    return img.cpu().numpy()


def _novel(state):
    """The VDI as a view-dependent volume: each view ray walked through the generating camera's pixel columns."""
    case, reg = state["case"], state["reg"]
    W, H, n_s = case["w"], case["h"], case["n_s"]
    g, v = state["cam"], state["view"]
    gc, vc = (_Cam(list(c.eye), list(c.center), W, H) for c in (g, v))
    fb, rgba = (x.double() for x in reg.records_f32())
    if case["prec"] == 1:
        raw = reg.rgba.view(W * H, n_s, 4)[..., 2:].contiguous().view(torch.float16).double()
        tau = raw[..., 3]
        A = -torch.expm1(-tau * math.log(2.0))
    else:
        A = rgba[..., 3]
        tau = -torch.log2(1 - A)
    tau = tau.clamp(max=1e7)  # an opaque record: any part of it is opaque
    f, r, u = _basis(gc)
    rays = _rays(vc)
    dot = lambda b, x: b[0] * x[0] + b[1] * x[1] + b[2] * x[2]  # noqa: E731
    D = [dot(b, rays) for b in (r, u, f)]
    q3 = [a - b for a, b in zip(vc.eye, gc.eye)]
    Q = [dot(b, q3) for b in (r, u, f)]
    ty = math.tan(math.radians(FOVY) / 2)
    tx = ty * W / H
    s_in, s_out = torch.zeros_like(D[0]), torch.full_like(D[0], math.inf)
    for A0, B0 in ((Q[0] + tx * Q[2], D[0] + tx * D[2]), (tx * Q[2] - Q[0], tx * D[2] - D[0]),
                   (ty * Q[2] - Q[1], ty * D[2] - D[1]), (Q[1] + ty * Q[2], D[1] + ty * D[2])):
        s0 = -A0 / B0
        s_in = torch.where(B0 > 0, torch.maximum(s_in, s0), s_in)
        s_out = torch.where(B0 > 0, s_out, torch.minimum(s_out, s0))
    out = torch.zeros((W * H, 4), dtype=torch.float64, device=DEV)
    live = (s_out > s_in).nonzero()[:, 0]
    D, s, s_out = [d[live] for d in D], s_in[live], s_out[live]
    star = -(Q[0] * D[0] + Q[1] * D[1] + Q[2] * D[2])
    rho = torch.sqrt(sum((Q[a] + star * D[a]) ** 2 for a in range(3)))
    su = torch.where(D[0] * Q[2] - Q[0] * D[2] > 0, 1, -1)
    sv = torch.where(D[1] * Q[2] - Q[1] * D[2] > 0, -1, 1)
    z = Q[2] + s * D[2]
    sm = torch.where(torch.isinf(s_out), s + 1, 0.5 * (s + s_out))
    zm = Q[2] + sm * D[2]
    x0 = torch.where(z > 0, (Q[0] + s * D[0]) / z, (Q[0] + sm * D[0]) / zm)
    y0 = torch.where(z > 0, (Q[1] + s * D[1]) / z, (Q[1] + sm * D[1]) / zm)
    iu = ((x0 / tx + 1) * 0.5 * W).floor().clamp(0, W - 1).long()
    iv = ((1 - y0 / ty) * 0.5 * H).floor().clamp(0, H - 1).long()
    C, T = torch.zeros((live.numel(), 3), dtype=torch.float64, device=DEV), torch.ones_like(s)
    for _ in range(W + H + 8):
        if not live.numel():
            break
        bu, bv = torch.where(su > 0, iu + 1, iu), torch.where(sv > 0, iv + 1, iv)
        bx, by = (2.0 * bu / W - 1) * tx, (1 - 2.0 * bv / H) * ty
        sx, sy = -(Q[0] - bx * Q[2]) / (D[0] - bx * D[2]), -(Q[1] - by * Q[2]) / (D[1] - by * D[2])
        inf = torch.full_like(s, math.inf)
        sx = torch.where((bu > 0) & (bu < W) & (Q[2] + sx * D[2] > 0), sx, inf)
        sy = torch.where((bv > 0) & (bv < H) & (Q[2] + sy * D[2] > 0), sy, inf)
        sn = torch.minimum(torch.minimum(sx, sy), s_out)
        near = (star > s) & (star < sn)
        cu, cv = (sx < s_out) & (sx <= sy) & ~near, (sy < s_out) & (sy <= sx) & ~near
        done = ~cu & ~cv & ~near
        sn = torch.maximum(torch.where(near, star, sn), s)
        p = iv * W + iu
        m = ((reg.counts[p] > 0) & (sn > s)).nonzero()[:, 0]
        if m.numel():
            pm, rm = p[m], rho[m, None]
            F, B = fb[pm, :, 0], fb[pm, :, 1]
            ua, ub = (s[m] - star[m]).abs(), (sn[m] - star[m]).abs()
            off = [torch.sqrt(((c - rm) * (c + rm)).clamp(min=0.0)) * (c > rm) for c in (F, B)]
            l = (torch.minimum(off[1], torch.maximum(ua, ub)[:, None]) -
                 torch.maximum(off[0], torch.minimum(ua, ub)[:, None])).clamp(min=0.0)
            ok = (torch.arange(n_s, device=DEV)[None, :] < reg.counts[pm, None]) & (B > F) & (A[pm] > 0)
            x = torch.where(ok, tau[pm] * l / torch.where(ok, B - F, torch.ones_like(F)), torch.zeros_like(F))
            x = torch.where((s[m] >= star[m])[:, None], x, x.flip(1))
            c = torch.where(ok[..., None], rgba[pm, :, :3] / A[pm].clamp(min=1e-300)[..., None], torch.zeros(1, dtype=torch.float64, device=DEV))
            c = torch.where((s[m] >= star[m])[:, None, None], c, c.flip(1))
            L = x.cumsum(dim=1)
            wgt = T[m, None] * torch.exp2(-(L - x)) * -torch.expm1(-x * math.log(2.0))
            C[m] += (wgt[..., None] * c).sum(dim=1)
            T[m] *= torch.exp2(-L[:, -1])
        iu, iv, s = iu + su * cu, iv + sv * cv, sn
        done = done | (iu < 0) | (iu >= W) | (iv < 0) | (iv >= H) | (s >= s_out)
        if bool(done.any()):
            out[live[done]] = torch.cat([C[done], 1 - T[done][:, None]], dim=-1)
            k = ~done
            live, s, s_out, star, rho, su, sv, iu, iv, C, T = (a[k] for a in (live, s, s_out, star, rho, su, sv, iu, iv, C, T))
            D = [d[k] for d in D]
    return out.cpu().numpy()


def _trained(case, seed):
    """One Adam step on the mean squared error, with the weights rounded to bfloat16 in the passes."""
    with open(CKPT, "rb") as f:
        raw = f.read()[24:]  # after the header: FP32 weights, their BF16 copy, Adam's moments, the step count
    buf = torch.frombuffer(bytearray(raw), dtype=torch.uint8)
    theta, m, v = (_part(buf, at).to(DEV).double() for at in (WEIGHTS, MOMENT1, MOMENT2))
    t = struct.unpack("<Q", raw[STEPS:STEPS + 8])[0] + 1
    w = theta.float().bfloat16().double().requires_grad_(True)
    x, y, valid = _rows(case["rows"], seed)
    n = valid.double().sum()
    a, at = [], 0
    for shape in ((64, 40), (64,), (64, 64), (64,), (64,), (1,)):
        a.append(w[at:at + math.prod(shape)].view(shape))
        at += math.prod(shape)
    h = torch.relu(torch.relu(x.double() @ a[0].t() + a[1]) @ a[2].t() + a[3])
    loss = (((h @ a[4] + a[5]) - y.double()) ** 2 * valid.double()).sum() / n
    loss.backward()
    m, v = 0.9 * m + 0.1 * w.grad, 0.999 * v + 0.001 * w.grad ** 2
    new = theta - 3e-4 * (m / (1 - 0.9 ** t)) / (torch.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
    return {"weights": new.cpu().numpy(), "moment1": m.cpu().numpy(), "moment2": v.cpu().numpy(), "loss": loss.detach().view(1).cpu().numpy()}


def exact(case, seed):
    case = _plain(case)
    kind = case["kind"]
    lists = {"counts": None, "gamma": None, "rgba": None}
    if case.get("prec") == 0:
        lists["fb"] = None
    if kind == "frame":
        return dict(lists, image=_dvr(case, seed))
    if kind == "composite":
        s = _prepare(case, seed)
        return dict(lists, image=_flat_lists(s["outs"], case["w"] * case["h"], case["n_s"], case["prec"]))
    if kind == "comp_batch":
        s = _prepare(case, seed)
        return [dict(lists, image=_flat_lists(ins, q["w"] * q["h"], q["n_s"], case["prec"])) for q, ins, _, _ in s["keep"]]
    if kind == "render":
        return {"image": _novel(_prepare(case, seed))}
    if kind == "train":
        return _trained(case, seed)
    return None
