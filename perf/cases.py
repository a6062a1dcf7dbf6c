"""Performance cases: the work a program has this library do, through its public calls.

listed()  named cases; draw(rng) gives more of the same ranges
prepare   the inputs (made from the seed on the GPU) and the volume, batch or server a program keeps
run       one pass through the public entry points; the outputs whole
work      bytes and operations of a pass that no implementation can do without
exact     the floating outputs in 64 bits, from plain torch (no code of this library beyond the encoder
          that made the compressed input)

Volumes come in the shapes of synth/recipes.py: sphere distance fields (one closed surface), six-octave gradient
noise (turbulent sheets everywhere) and a channel-flow-like field (a mean profile with fluctuations), each written
here as a few matrix products so that making one takes milliseconds.
"""
import math

import numpy as np
import torch

import paper_2009_03254_gb300 as bc

LIGHT = (0.3, -0.5, 0.8)


def listed():
    return [
        # a small closed surface looked at again and again (an interactive view of a 64^3 region, 16 bits a value):
        # nothing to decode, so launches and latency are the whole call
        {"name": "sphere64_warm", "kind": "surface", "field": "sphere", "nx": 64, "ny": 64, "nz": 64, "rate": 16,
         "isos": 1, "cold": False, "format": "float4"},
        # the benchmark's workload: a Plasma-sized 512^3 volume at 8 bits a value, five isovalues from an empty cache
        {"name": "noise512_sweep", "kind": "surface", "field": "noise", "nx": 512, "ny": 512, "nz": 512, "rate": 8,
         "isos": 5, "cold": True, "format": "float4"},
        # a scan of odd size at 11 bits a value, its surface in the paper's compact 8-byte vertices, from an empty cache
        {"name": "ragged_packed", "kind": "surface", "field": "noise", "nx": 397, "ny": 301, "nz": 259, "rate": 11,
         "isos": 1, "cold": True, "format": "packed"},
        # an indexed mesh for a consumer that shares vertices, blocks already cached (a slider moved over two values)
        {"name": "indexed_warm", "kind": "surface", "field": "channel", "nx": 320, "ny": 256, "nz": 384, "rate": 12,
         "isos": 2, "cold": False, "format": "indexed"},
        # the largest: a 1024^3 channel flow at 4 bits a value, its first surface
        {"name": "channel1024", "kind": "surface", "field": "channel", "nx": 1024, "ny": 1024, "nz": 1024, "rate": 4,
         "isos": 1, "cold": True, "format": "float4"},
        # many small volumes at once (32 to 256 a side, 8 to 16 bits a value), one surface each
        {"name": "batch64", "kind": "batch", "count": 64, "lo": 32, "hi": 256},
        # a service answering queued isovalue requests on one resident volume
        {"name": "serve_channel", "kind": "serve", "nx": 512, "ny": 384, "nz": 256, "rate": 2, "requests": 8,
         "max_batch": 4},
        # a time series: each step arrives compressed in pinned host memory, one surface of it, then it is dropped
        {"name": "load_extract", "kind": "load", "field": "noise", "nx": 257, "ny": 322, "nz": 288, "rate": 8},
        # full decompression, the baseline of the paper's comparison and what a consumer of samples asks for
        {"name": "decode512", "kind": "decode", "field": "noise", "nx": 512, "ny": 512, "nz": 512, "rate": 8},
        # compressing a simulation's field of odd size
        {"name": "encode_ragged", "kind": "encode", "field": "channel", "nx": 499, "ny": 333, "nz": 218, "rate": 6},
        # drawing an extracted surface at 1080p
        {"name": "render1080", "kind": "render", "field": "noise", "nx": 512, "ny": 512, "nz": 512, "rate": 8,
         "width": 1920, "height": 1080, "format": "float4"},
        # the same kind of view ray cast from the block cache
        {"name": "raycast1080", "kind": "raycast", "field": "noise", "nx": 512, "ny": 512, "nz": 512, "rate": 8,
         "width": 1920, "height": 1080},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def dims(lo, hi):
        return {"nx": log_int(lo, hi), "ny": log_int(lo, hi), "nz": log_int(lo, hi)}

    kind = rng.choice(["surface"] * 5 + ["batch", "serve", "load", "decode", "encode", "render", "raycast"])
    field = rng.choice(["sphere", "noise", "channel"])
    if kind == "surface":
        return {"kind": kind, "field": field, **dims(32, 768), "rate": rng.randint(2, 16), "isos": rng.randint(1, 5),
                "cold": rng.random() < 0.5, "format": rng.choice(["float4", "float4", "packed", "indexed", "indexed_packed"])}
    if kind == "batch":
        lo = log_int(24, 64)
        return {"kind": kind, "count": log_int(2, 96), "lo": lo, "hi": lo * rng.randint(2, 4)}
    if kind == "serve":
        return {"kind": kind, **dims(128, 768), "rate": rng.randint(2, 8), "requests": rng.randint(1, 12),
                "max_batch": rng.randint(1, 8)}
    if kind == "load":
        return {"kind": kind, "field": field, **dims(48, 512), "rate": rng.randint(2, 16)}
    if kind in ("decode", "encode"):
        return {"kind": kind, "field": field, **dims(32, 640), "rate": rng.randint(1, 24)}
    w = log_int(256, 2560)
    view = {"kind": kind, "field": field, **dims(48, 512), "rate": rng.randint(4, 12), "width": w,
            "height": max(1, int(w * rng.uniform(0.4, 1.0)))}
    if kind == "render":
        view["format"] = rng.choice(["float4", "packed", "indexed"])
    return view


# ---------------------------------------------------------------- inputs

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _octave(dims, period, gen):
    """Gradient noise of one lattice period: sum over lattice points of (gradient . offset) times the quintic fade
    weights, which separates into one small matrix per axis."""
    grads = torch.tensor([(a, b, 0) for a in (1, -1) for b in (1, -1)] + [(a, 0, b) for a in (1, -1) for b in (1, -1)] +
                         [(0, a, b) for a in (1, -1) for b in (1, -1)], dtype=torch.float32, device="cuda")
    weight, offset = [], []
    for n in dims:
        x = torch.arange(n, device="cuda", dtype=torch.float32) / period
        cell = torch.floor(x)
        f = x - cell
        fade = f * f * f * (f * (f * 6.0 - 15.0) + 10.0)
        rows, c = torch.arange(n, device="cuda"), cell.long()
        w = torch.zeros((n, (n - 1) // period + 2), device="cuda")
        d = torch.zeros_like(w)
        w[rows, c], w[rows, c + 1] = 1.0 - fade, fade
        d[rows, c], d[rows, c + 1] = (1.0 - fade) * f, fade * (f - 1.0)
        weight.append(w)
        offset.append(d)
    lx, ly, lz = (w.shape[1] for w in weight)
    g = grads[torch.randint(0, 12, (lz, ly, lx), generator=gen, device="cuda")]
    out = None
    for axis in range(3):
        mx, my, mz = (offset[k] if k == axis else weight[k] for k in range(3))
        t = g[..., axis] @ mx.T                                          # (lz, ly, nx)
        t = torch.matmul(my, t)                                          # (lz, ny, nx)
        t = mz @ t.reshape(lz, -1)                                       # (nz, ny * nx)
        out = t if out is None else out.add_(t)
    return out.view(dims[2], dims[1], dims[0])


def _noise(dims, gen, octaves, base, gain):
    f = torch.zeros((dims[2], dims[1], dims[0]), device="cuda")
    for o in range(octaves):
        f.add_(_octave(dims, base >> o, gen), alpha=3.0 * gain ** o)
    return f


def _rank(f, p):
    """the value at rank p of the field (of every some-th sample)"""
    v = torch.sort(f.view(-1)[:: max(1, f.numel() >> 18)]).values
    return float(v[min(v.numel() - 1, int(p * v.numel()))])


def _field(kind, dims, seed):
    """(field (nz, ny, nx), the isovalues of its surfaces as a function of how many are wanted)"""
    gen = _generator(seed)
    if kind == "sphere":
        r = 0.3125 * min(dims)
        jitter = torch.rand(3, generator=gen, device="cuda") * 0.1 * r
        sq = [(torch.arange(n, device="cuda", dtype=torch.float32) - ((n - 1) / 2 + jitter[k])) ** 2 for k, n in enumerate(dims)]
        f = torch.sqrt(sq[0][None, None, :] + sq[1][None, :, None] + sq[2][:, None, None]) - r
        return f.contiguous(), lambda n: [0.1 * r * (k - (n - 1) / 2) / max(n, 1) for k in range(n)]
    if kind == "noise":
        f = _noise(dims, gen, 6, 128, 0.5)
        return f, lambda n: [_rank(f, 0.5 + 0.34 * (2 * k / (n - 1) - 1 if n > 1 else 0)) for k in range(n)]   # +- 1 deviation
    z = torch.arange(dims[2], device="cuda", dtype=torch.float64) / max(dims[2] - 1, 1)
    u = torch.tanh(z / 0.08) * torch.tanh((1.0 - z) / 0.08)
    f = _noise(dims, gen, 7, 256, 2.0 ** (-1.0 / 3.0))
    f.mul_((0.3 * (1.0 - u) + 0.1).float()[:, None, None]).add_(u.float()[:, None, None])
    return f, lambda n: [_rank(f, 0.7 - 0.1 * k) for k in range(n)]


def _dims(case):
    return case["nx"], case["ny"], case["nz"]


def _compressed(case, seed, kind=None):
    """(compressed volume, isovalues): (bits, block minima, block maxima) on the device"""
    f, isos = _field(kind or case["field"], _dims(case), seed)
    return bc.encode_field(f, case["rate"]), isos


def _batch_members(case, seed):
    rng = np.random.default_rng(int(seed))
    members = []
    for i in range(case["count"]):
        d = [int(round(math.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]))))) for _ in range(3)]
        members.append({"nx": d[0], "ny": d[1], "nz": d[2], "rate": int(rng.integers(8, 17)),
                        "field": ("sphere", "noise")[int(rng.integers(2))], "seed": int(rng.integers(1 << 30))})
    return members


def _batch_room(case):
    return int(case["count"] * 0.12 * (case["lo"] * case["hi"]) ** 1.5) + 65536


def _serve_isos(case, seed, isos):
    """a walk over the middle of the value range, as neighbouring requests of a session come"""
    rng = np.random.default_rng(int(seed))
    at, got = 3.0, []
    for _ in range(case["requests"]):
        at = min(6.0, max(0.0, at + rng.uniform(-1.0, 1.0)))
        got.append(float(isos(1)[0]) + 0.02 * (at - 3.0))
    return got


def _camera(dims, seed):
    """(eye, forward, right, up) of a view from outside onto the whole volume, 45 degrees high"""
    rng = np.random.default_rng(int(seed))
    az, el = np.radians(rng.uniform(0, 360)), np.radians(rng.uniform(10, 40))
    c, r = np.asarray(dims, float) / 2, 1.6 * float(np.linalg.norm(dims))
    eye = c + r * np.array([np.cos(el) * np.cos(az), np.cos(el) * np.sin(az), np.sin(el)])
    fwd = (c - eye) / np.linalg.norm(c - eye)
    right = np.cross(fwd, (0.0, 0.0, 1.0))
    right /= np.linalg.norm(right)
    return eye, fwd, right, np.cross(right, fwd), r


def _view_proj(dims, seed, aspect):
    eye, fwd, right, up, r = _camera(dims, seed)
    t, near, far = 1.0 / math.tan(math.radians(22.5)), 0.05 * r, 3.0 * r
    proj = np.array([[t / aspect, 0, 0, 0], [0, t, 0, 0],
                     [0, 0, (far + near) / (near - far), 2 * far * near / (near - far)], [0, 0, -1, 0]])
    view = np.eye(4)
    view[:3, :3] = np.stack([right, up, -fwd])
    view[:3, 3] = -view[:3, :3] @ eye
    return (proj @ view).astype(np.float32)


def _volume(case, bits, bmin, bmax):
    return bc.Volume(bits, _dims(case), case["rate"], bmin, bmax)


def _room(field, dims):
    """triangles that a surface of the field above has at most, with some to spare: what the caller's buffers hold"""
    samples = math.prod(dims)
    if field == "sphere":
        return int(5 * 4 * math.pi * (0.3125 * min(dims)) ** 2) + 4096
    return int((0.12 if field == "noise" else 0.32) * samples) + 4096


def _buffers(vol, field, dims, isos, fmt):
    """a zeroed buffer per surface, kept and written again and again; an extraction without room tells a surface's size"""
    got = []
    for iso in isos:
        t = vol.extract_into(iso, torch.empty((0, 4), device="cuda"), check=False)["num_triangles"]
        t = max(t, _room(field, dims))
        if fmt.startswith("indexed"):          # at most about 0.8 vertices a triangle, except on the smallest
            n = t + 64
            got.append((torch.zeros((n, 2), dtype=torch.int32, device="cuda") if fmt.endswith("packed")
                        else torch.zeros((n, 4), device="cuda"), torch.zeros((t, 3), dtype=torch.int32, device="cuda")))
        else:
            got.append(torch.zeros((3 * t, 2), dtype=torch.int32, device="cuda") if fmt == "packed"
                       else torch.zeros((3 * t, 4), device="cuda"))
    return got


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        vols, isos = [], []
        for m in _batch_members(case, seed):
            (bits, lo, hi), of = _compressed(m, m["seed"])
            vols.append(_volume(m, bits, lo, hi))
            isos.append(of(1)[0])
        batch = bc.Batch(vols)
        isos = np.asarray(isos, np.float32)
        total = max(_batch_room(case), int(batch.extract_into(isos, None, check=False)["offsets"][-1]))
        return {"kind": kind, "batch": batch, "vols": vols, "isos": isos,
                "out": torch.zeros((3 * total, 4), device="cuda")}
    if kind == "encode":
        f, _ = _field(case["field"], _dims(case), seed)
        nb = int(np.prod(bc.block_dims(_dims(case))))
        out = (torch.empty((nb, case["rate"]), dtype=torch.int64, device="cuda"), torch.empty(nb, device="cuda"),
               torch.empty(nb, device="cuda"))
        return {"kind": kind, "field": f, "rate": case["rate"], "out": out}
    (bits, lo, hi), of = _compressed(case, seed, "channel" if kind == "serve" else None)
    if kind == "decode":
        return {"kind": kind, "bits": bits, "dims": _dims(case), "rate": case["rate"],
                "out": torch.empty((case["nz"], case["ny"], case["nx"]), device="cuda")}
    if kind == "load":
        host = [t.cpu().pin_memory() for t in (bits, lo, hi)]
        vol = _volume(case, bits, lo, hi)
        out = _buffers(vol, case["field"], _dims(case), of(1), "float4")[0]
        vol.release()
        return {"kind": kind, "host": host, "dims": _dims(case), "rate": case["rate"], "iso": of(1)[0], "out": out}
    vol = _volume(case, bits, lo, hi)
    if kind == "serve":
        isos = _serve_isos(case, seed, of)
        return {"kind": kind, "vol": vol, "server": bc.Server(vol, max_batch=case["max_batch"], packed=True),
                "isos": isos, "out": _buffers(vol, "channel", _dims(case), isos, "packed")}
    if kind == "surface":
        isos = of(case["isos"])
        return {"kind": kind, "vol": vol, "isos": isos, "cold": case["cold"], "format": case["format"],
                "out": _buffers(vol, case["field"], _dims(case), isos, case["format"])}
    view = {"kind": kind, "dims": _dims(case), "width": case["width"], "height": case["height"],
            "rgba": torch.empty((case["height"], case["width"]), dtype=torch.int32, device="cuda"),
            "depth": torch.empty((case["height"], case["width"]), dtype=torch.int64, device="cuda")}
    aspect = case["width"] / case["height"]
    if kind == "raycast":
        eye, fwd, right, up, _ = _camera(_dims(case), seed)
        h = math.tan(math.radians(22.5))
        return {**view, "vol": vol, "iso": of(1)[0], "camera": (eye, fwd, right * h * aspect, up * h)}
    out = _buffers(vol, case["field"], _dims(case), of(1), case["format"])[0]
    if case["format"] == "indexed":
        tris = vol.extract_indexed_into(of(1)[0], *out)["num_triangles"]
    elif case["format"] == "packed":
        tris = vol.extract_packed_into(of(1)[0], out)["num_triangles"]
    else:
        tris = vol.extract_into(of(1)[0], out)["num_triangles"]
    vol.release()
    verts, idx = out if case["format"] == "indexed" else (out, None)
    return {**view, "verts": verts, "idx": idx, "tris": tris, "view_proj": _view_proj(_dims(case), seed, aspect)}


# ---------------------------------------------------------------- a pass

def _soup(v):
    """positions and block ids of float4 vertices"""
    return {"positions": v[:, :3], "blocks": v.view(torch.int32)[:, 3]}


def run(state):
    kind = state["kind"]
    if kind == "surface":
        vol, fmt = state["vol"], state["format"]
        if state["cold"]:
            vol.cache_reset()
        got = []
        for iso, out in zip(state["isos"], state["out"]):
            if fmt == "float4":
                vol.extract_into(iso, out)
                got.append(_soup(out))
            elif fmt == "packed":
                vol.extract_packed_into(iso, out)
                got.append(out)
            else:
                vol.extract_indexed_into(iso, *out)
                got.append({**(_soup(out[0]) if fmt == "indexed" else {"codes": out[0]}), "indices": out[1]})
        return got
    if kind == "batch":
        r = state["batch"].extract_into(state["isos"], state["out"])
        return {**_soup(state["out"]), "offsets": r["offsets"].astype(np.int64)}
    if kind == "serve":
        server = state["server"]
        tickets = [server.submit(iso) for iso in state["isos"]]
        while server.queued():
            server.step()
        for ticket, out in zip(tickets, state["out"]):       # each answer goes where its client reads it
            mesh = server.take(ticket)[1]
            out[:3 * mesh.num_triangles].copy_(mesh.vertices)
            mesh.release()
        return state["out"]
    if kind == "load":
        bits, lo, hi = state["host"]
        vol = bc.Volume(bits, state["dims"], state["rate"], lo, hi, async_upload=True)
        vol.extract_into(state["iso"], state["out"])
        vol.release()
        return _soup(state["out"])
    if kind == "decode":
        return bc.decode_volume(state["bits"], state["dims"], state["rate"], out=state["out"])
    if kind == "encode":
        bits, lo, hi = bc.encode_field(state["field"], state["rate"], out=state["out"])
        return {"bits": bits, "lo": lo, "hi": hi}
    if kind == "raycast":
        hits, rgba, st = state["vol"].raycast(state["iso"], *state["camera"], LIGHT, state["width"], state["height"],
                                              hits=state["depth"], rgba=state["rgba"])
        return {"hits": hits, "rgba": rgba, "count": st["hits"]}
    frag, rgba, _ = bc.render(state["verts"], state["tris"], state["dims"], state["view_proj"], LIGHT, state["width"],
                              state["height"], indices=state["idx"], fragments=state["depth"], rgba=state["rgba"])
    return {"fragments": frag, "rgba": rgba}


# ---------------------------------------------------------------- what a pass cannot do without

# measured shares of active blocks and triangles a sample of the fields above (mean over their isovalues and seeds)
_DENSITY = {"noise": (0.32, 0.070), "channel": (0.62, 0.22)}


def _counts(field, dims):
    """(blocks, active blocks, triangles) of one surface, about"""
    nb = math.prod((n + 3) // 4 for n in dims)
    if field == "sphere":                          # a closed surface: its area decides
        area = 4 * math.pi * (0.3125 * min(dims)) ** 2
        return nb, min(nb, area / 4), 3.0 * area
    act, tri = _DENSITY[field]
    return nb, act * nb, tri * math.prod(dims)


def _surface_work(field, dims, rate, isos, cold, tri_bytes=48):
    """ranges of every block and the active blocks' samples (compressed when the cache starts empty, else the decoded
    ones) in, triangles out; of a sweep's active blocks about a third are new at each isovalue after the first"""
    nb, act, tri = _counts(field, dims)
    new = act * (1 + (isos - 1) / 3) if cold else 0
    read = 8 * rate * new + 256 * (act * isos - new)
    return {"bytes": isos * (8 * nb + tri_bytes * tri) + read, "flops": isos * 36 * tri + new * 64 * 12}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        side = math.log(case["hi"] / case["lo"])
        mean = (case["hi"] - case["lo"]) / side if side else case["lo"]       # of a log-uniform side
        parts = [_surface_work(f, (mean,) * 3, 12, 1, False) for f in ("sphere", "noise")]
        return {k: case["count"] / 2 * sum(p[k] for p in parts) for k in ("bytes", "flops")}
    dims, samples = _dims(case), case["nx"] * case["ny"] * case["nz"]
    nb = math.prod((n + 3) // 4 for n in dims)
    if kind == "surface":
        tri_bytes = {"float4": 48, "packed": 24, "indexed": 25, "indexed_packed": 18}[case["format"]]
        return _surface_work(case["field"], dims, case["rate"], case["isos"], case["cold"], tri_bytes)
    if kind == "serve":
        w = _surface_work("channel", dims, case["rate"], case["requests"], False, 24)
        return {"bytes": w["bytes"] + case["requests"] * 48 * _DENSITY["channel"][1] * samples, "flops": w["flops"]}
    if kind == "load":
        w = _surface_work(case["field"], dims, case["rate"], 1, True)
        return {"bytes": w["bytes"] + 8 * case["rate"] * nb, "flops": w["flops"]}
    if kind in ("decode", "encode"):
        return {"bytes": 4 * samples + 8 * case["rate"] * nb + (8 * nb if kind == "encode" else 0), "flops": 12 * samples}
    pixels = case["width"] * case["height"]
    _, act, tri = _counts(case["field"], dims)
    if kind == "render":
        return {"bytes": {"float4": 48, "packed": 24, "indexed": 25}[case["format"]] * tri + 12 * pixels, "flops": 100 * tri}
    return {"bytes": 12 * pixels + 8 * nb + 256 * 0.1 * act, "flops": 400 * pixels}


# ---------------------------------------------------------------- the outputs in 64 bits

def _window(words, base, pos):
    """64 bits of each block's stream from bit `pos` on, as int64"""
    w = base + (pos >> 6)
    s = pos & 63
    lo, hi = words[w], words[w + 1]
    rest = torch.where(s == 0, -1, (torch.ones_like(s) << (64 - s).clamp(max=62)) - 1)
    rest = torch.where(s == 1, torch.full_like(s, (1 << 63) - 1), rest)
    return ((lo >> s) & rest) | torch.where(s == 0, 0, hi << (64 - s).clamp(max=63))


def _low(n):
    """a mask of the n lowest bits, n in 0..64"""
    return torch.where(n >= 64, -1, torch.where(n == 63, (1 << 63) - 1, (torch.ones_like(n) << n.clamp(max=62)) - 1))


def _decode(bits, rate, rounded):
    """The samples (nb, 64) of compressed blocks: the stream format that include/bcmc.h refers to, block by block in
    step.  `rounded`: each integer rounded to float32 before its scale, as the format has it."""
    out = torch.empty((bits.shape[0], 64), dtype=torch.float32 if rounded else torch.float64, device="cuda")
    seq = [0, 1, 2, 2]
    coded = sorted(range(64), key=lambda l: (seq[l & 3] + seq[l >> 2 & 3] + seq[l >> 4], l))
    for b0 in range(0, bits.shape[0], 1 << 21):
        part = bits[b0:b0 + (1 << 21)]
        nb = part.shape[0]
        words = torch.cat([part.reshape(-1), torch.zeros(2, dtype=torch.int64, device="cuda")])
        base = torch.arange(nb, device="cuda") * rate
        head = part[:, 0]
        live0 = (head & 1) == 1
        e = ((head >> 1) & 255) - 127
        end = torch.where(live0, 64 * rate, 0)
        pos = torch.full_like(base, 9)
        n = torch.zeros_like(base)
        coef = [torch.zeros(nb, dtype=torch.int64, device="cuda") for _ in range(64)]
        for k in range(31, -1, -1):
            m = torch.minimum(n, (end - pos).clamp(min=0))
            plane = _window(words, base, torch.minimum(pos, end)) & _low(m)
            pos = pos + m
            at = torch.nonzero((pos < end) & (n < 64)).view(-1)
            while at.numel():
                p, r, b, stop = pos[at], n[at], base[at], end[at]
                some = (_window(words, b, p) & 1) == 1
                p = p + 1
                limit = 63 - r
                scan = torch.minimum(limit, stop - p)
                w = _window(words, b, torch.minimum(p, stop)) & _low(scan)
                zeros = torch.log2((w & -w).double().clamp(min=1)).round().long()
                found = some & (w != 0)
                last = some & (w == 0) & (scan == limit)
                cut = some & (w == 0) & (scan < limit)
                bit = torch.where(last, 63, r + zeros)
                plane[at] = torch.where(found | last, plane[at] | (torch.ones_like(bit) << bit.clamp(0, 63)), plane[at])
                n[at] = torch.where(found, r + zeros + 1, torch.where(last, 64, r))
                p = torch.where(found, p + zeros + 1, torch.where(last, p + limit, torch.where(cut, stop, p)))
                pos[at] = p
                at = at[some & (p < stop) & (n[at] < 64)]
            for i in range(64):
                coef[i] |= ((plane >> i) & 1) << k
        mask = 0xAAAAAAAA
        q = [None] * 64
        for i, l in enumerate(coded):
            q[l] = (((coef[i] ^ mask) - mask) & 0xFFFFFFFF).to(torch.int32)
        for step in (16, 4, 1):
            for l in range(64):
                if (l // step) & 3:
                    continue
                ll, hh, h0, h1 = (q[l + step * j] for j in range(4))
                l1 = ll - (hh >> 1)
                l0 = hh + l1
                b = l0 - (h0 >> 1)
                d = l1 - (h1 >> 1)
                q[l], q[l + step], q[l + 2 * step], q[l + 3 * step] = h0 + b, b, h1 + d, d
        scale = torch.exp2((e - 27).double())
        for l in range(64):
            v = (q[l].float().double() if rounded else q[l].double()) * scale
            out[b0:b0 + nb, l] = torch.where(live0, v, 0.0)
    return out


def _dense(samples, dims):
    nbx, nby, nbz = bc.block_dims(dims)
    f = samples.view(nbz, nby, nbx, 4, 4, 4).permute(0, 3, 1, 4, 2, 5).reshape(4 * nbz, 4 * nby, 4 * nbx)
    return f[:dims[2], :dims[1], :dims[0]].contiguous()


def _case_table():
    """triangles (up to 5, as edge numbers) of the 256 cell cases: on every face each run of corners below the
    isovalue is cut off by one segment, the segments link into cycles, each fanned from its smallest edge"""
    def edge(c, d):
        axis, low = {1: 0, 2: 1, 4: 2}[c ^ d], min(c, d)
        rest = [low >> a & 1 for a in range(3) if a != axis]
        return 4 * axis + rest[0] + 2 * rest[1]

    table = []
    for case in range(256):
        below = [bool(case >> c & 1) for c in range(8)]
        follow = {}
        for a in range(3):
            b, c = (a + 1) % 3, (a + 2) % 3
            for side in (0, 1):
                ring = [(side << a) | (u << b) | (v << c) for u, v in ((0, 0), (1, 0), (1, 1), (0, 1))]
                ring = ring if side else ring[:1] + ring[:0:-1]
                for i in range(4):
                    if not below[ring[i - 1]] and below[ring[i]]:
                        j = i
                        while below[ring[(j + 1) % 4]]:
                            j += 1
                        follow[edge(ring[i - 1], ring[i])] = edge(ring[j % 4], ring[(j + 1) % 4])
        tris = []
        while follow:
            e = min(follow)
            cycle = []
            while e in follow:
                cycle.append(e)
                e = follow.pop(e)
            tris += [(cycle[0], cycle[k], cycle[k + 1]) for k in range(1, len(cycle) - 1)]
        table.append(tris)
    return table


def _surface(field, iso):
    """(positions (3T, 3) in 64 bits and a key per vertex: its block, then edge inside it) in block order"""
    nz, ny, nx = field.shape
    nbx, nby, _ = bc.block_dims((nx, ny, nz))
    if min(nx, ny, nz) < 2:
        return torch.empty((0, 3), dtype=torch.float64, device="cuda"), torch.empty(0, dtype=torch.int64, device="cuda")
    iso = float(np.float32(iso))
    low = field < iso
    case = torch.zeros((nz - 1, ny - 1, nx - 1), dtype=torch.uint8, device="cuda")
    for c in range(8):
        i, j, k = c & 1, c >> 1 & 1, c >> 2
        case |= low[k:nz - 1 + k, j:ny - 1 + j, i:nx - 1 + i].to(torch.uint8) << c
    flat = case.view(-1)
    cell = torch.nonzero((flat != 0) & (flat != 255)).view(-1)
    x, y, z = cell % (nx - 1), cell // (nx - 1) % (ny - 1), cell // ((nx - 1) * (ny - 1))
    block = (x >> 2) + nbx * ((y >> 2) + nby * (z >> 2))
    order = torch.argsort(block * 64 + (x & 3) + 4 * (y & 3) + 16 * (z & 3))
    cs, x, y, z, block = flat[cell[order]].long(), x[order], y[order], z[order], block[order]
    table = _case_table()
    count = torch.tensor([len(t) for t in table], device="cuda")[cs]
    rows = torch.tensor([[e for t in tris for e in t] + [0] * (15 - 3 * len(tris)) for tris in table], device="cuda")
    at = torch.repeat_interleave(torch.arange(cs.numel(), device="cuda"), 3 * count)
    first = torch.cumsum(3 * count, 0) - 3 * count
    e = rows[cs[at], torch.arange(at.numel(), device="cuda") - first[at]]
    axis, m = e >> 2, e & 3
    step = [(axis == a).long() for a in range(3)]
    dx = torch.where(axis == 0, 0, m & 1)
    dy = torch.where(axis == 0, m & 1, torch.where(axis == 1, 0, m >> 1))
    dz = torch.where(axis == 2, 0, m >> 1)
    px, py, pz = x[at] + dx, y[at] + dy, z[at] + dz
    f = field.view(-1)
    v0 = f[px + nx * (py + ny * pz)].double()
    v1 = f[px + step[0] + nx * (py + step[1] + ny * (pz + step[2]))].double()
    t = (iso - v0) / (v1 - v0)
    corner = [(x[at] & 3) + dx, (y[at] & 3) + dy, (z[at] & 3) + dz]
    pos = torch.stack([corner[a].double() + step[a] * t for a in range(3)], 1)
    return pos, block[at] * 512 + axis * 125 + corner[0] + 5 * corner[1] + 25 * corner[2]


def _surface_positions(field, iso, room, indexed=False):
    """as _soup() of a zeroed buffer with room for so many triangles"""
    pos, key = _surface(field, iso)
    tris = max(room, pos.shape[0] // 3)
    out = torch.zeros((tris + 64 if indexed else 3 * tris, 3), dtype=torch.float64, device="cuda")
    if indexed:                                    # one vertex per block and cut edge, in that order
        out[torch.unique(key, return_inverse=True)[1]] = pos
    else:
        out[:pos.shape[0]] = pos
    return {"positions": out, "blocks": None, **({"indices": None} if indexed else {})}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("serve", "encode", "render", "raycast") or "packed" in case.get("format", ""):
        return None                                # whole numbers, or ranges of what the encoder wrote
    if kind == "batch":
        if case["count"] * (case["lo"] * case["hi"]) ** 1.5 > 4e8:
            return None
        parts = []
        for m in _batch_members(case, seed):
            (bits, _, _), of = _compressed(m, m["seed"])
            iso = of(1)[0]
            parts.append(_surface(_dense(_decode(bits, m["rate"], True), _dims(m)), iso)[0])
        pos = torch.cat(parts)
        out = torch.zeros((max(3 * _batch_room(case), pos.shape[0]), 3), dtype=torch.float64, device="cuda")
        out[:pos.shape[0]] = pos
        return {"positions": out, "blocks": None, "offsets": None}
    if math.prod(_dims(case)) > 1.5e8:
        return None
    (bits, _, _), of = _compressed(case, seed)
    if kind == "decode":
        return _dense(_decode(bits, case["rate"], False), _dims(case))
    field, room = _dense(_decode(bits, case["rate"], True), _dims(case)), _room(case["field"], _dims(case))
    if kind == "load":
        return _surface_positions(field, of(1)[0], room)
    return [_surface_positions(field, iso, room, case["format"] == "indexed") for iso in of(case["isos"])]
