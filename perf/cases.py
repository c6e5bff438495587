"""Workloads of the steganography library, each run through its public entry points.

A case is one of five kinds of use:

  still   one image: hide a message in it, optionally measure the change (the count and squared error behind
          PSNR), and read the message back.  Any layout of the library (one bit per byte, k bits, one colour
          plane, the paper's two-bit plane layout), images of any size, buffers at any address (a frame of a
          packed stack starts wherever the frames before it end).
  batch   many covers of different sizes, in one batched call per direction.
  video   the frames of one video, back to back in memory, a captured batched call per direction.
  serve   a burst of mixed requests to a server: submit, wait, collect.
  host    a batch of covers in pinned host memory through the host pipeline.

Pixels and messages are uniform random bytes (compressed or encrypted messages are), video frames a smooth
gradient with noise.
"""
import math
import random

import numpy as np
import torch

import paper_0912_0947_gb300 as S

HEADER_BYTES = 4  # the stream layout's length field


def _still(name, w, h, ch, **more):
    c = {"name": name, "kind": "still", "w": w, "h": h, "ch": ch, "layout": "stream", "k": 1, "plane": -1,
         "header": True, "fill": 1.0, "cover_at": 0, "stego_at": 0, "msg_at": 0, "inplace": False,
         "stats": True, "quality": False}
    c.update(more)
    return c


def _batch(name, count, lo, hi, **more):
    c = {"name": name, "kind": "batch", "count": count, "lo": lo, "hi": hi, "mix": 1, "layout": "stream",
         "align": 256}
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: one web-sized image with a short text, where latency and launches count
        _still("still_small", 512, 512, 3, fill=1 / 3),
        # the largest still: a scan filled to capacity
        _still("still_full", 8192, 8192, 3),
        # an odd-sized frame taken out of a packed stack (its first byte lies anywhere), written to a buffer
        # of its own, checked against the original, and read back
        _still("still_ragged", 3839, 2159, 3, fill=0.7, cover_at=13, stats=False, quality=True),
        # a camera picture with two bits in every byte: twice the payload
        _still("still_k2", 6000, 4000, 3, k=2, fill=0.9),
        # three bits in the green plane only, image and output both views into packed stacks
        _still("plane_ragged_k3", 3839, 2159, 3, k=3, plane=1, fill=0.8, cover_at=13, stego_at=13, msg_at=5),
        # the paper's own layout on a picture whose rows are not whole 16-byte vectors
        _still("paper_odd", 5471, 3647, 3, layout="paper", plane=0, header=False, fill=0.9),
        # a few thumbnails and web images in one call: what a lightly loaded service has in hand
        _batch("batch_small", 16, 64, 512),
        # thousands of covers of every size, the throughput case
        _batch("batch_uneven", 4096, 64, 4096),
        # the same mix of sizes in the paper's layout
        _batch("batch_paper", 1024, 64, 4096, layout="paper"),
        # 600 full-HD frames at half capacity, replayed as a captured graph
        {"name": "video_hd", "kind": "video", "w": 1920, "h": 1080, "frames": 600, "layout": "stream",
         "fill": 0.5},
        # a burst of mixed requests, 70% to embed and 30% to extract
        {"name": "serve_burst", "kind": "serve", "count": 2048, "lo": 64, "hi": 4096, "mix": 1},
        # covers that live in host memory, with a read-back check of every stego
        {"name": "host_batch", "kind": "host", "count": 96, "lo": 64, "hi": 4096, "mix": 1},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["still", "batch", "video", "serve", "host"], [10, 5, 2, 1, 1])[0]
    if kind == "still":
        w, h = _log(rng, 64, 8192), _log(rng, 64, 8192)
        if rng.random() < 0.4:
            w = max(64, w // 16 * 16)  # the widths that cameras and screens have
        ch = rng.choice([1, 3, 3, 3, 4])
        paper = rng.random() < 0.35
        plane = rng.randrange(ch) if paper or rng.random() < 0.35 else -1
        inplace = rng.random() < 0.2
        cover_at = rng.choice([0, 0, rng.randrange(1, 16)])
        c = _still("", w, h, ch, layout="paper" if paper else "stream", k=1 if paper else rng.choice([1, 1, 2, 3, 4]),
                   plane=plane, header=not paper and rng.random() < 0.8, fill=rng.uniform(0.05, 1.0),
                   cover_at=cover_at, stego_at=cover_at if inplace else rng.choice([0, cover_at]),
                   msg_at=rng.choice([0, 0, rng.randrange(1, 16)]), inplace=inplace,
                   stats=rng.random() < 0.7, quality=not inplace and rng.random() < 0.3)
    elif kind == "batch":
        paper = rng.random() < 0.4
        c = _batch("", _log(rng, 1, 512 if paper else 2048), 64, _log(rng, 128, 4096), mix=rng.randrange(1 << 20),
                   layout="paper" if paper else "stream", align=rng.choice([256, 256, 1]))
    elif kind == "video":
        c = {"kind": "video", "w": rng.choice([640, 854, 1280, 1366, 1920, 1080]), "h": rng.choice([360, 480, 720, 1080]),
             "frames": _log(rng, 8, 300), "layout": rng.choice(["stream", "paper"]), "fill": rng.uniform(0.05, 1.0)}
    elif kind == "serve":
        c = {"kind": "serve", "count": _log(rng, 8, 1024), "lo": 64, "hi": _log(rng, 128, 4096),
             "mix": rng.randrange(1 << 20)}
    else:
        c = {"kind": "host", "count": _log(rng, 4, 64), "lo": 64, "hi": _log(rng, 256, 4096),
             "mix": rng.randrange(1 << 20)}
    c.pop("name", None)
    return c


# -- sizes ---------------------------------------------------------------------


def _covers(case):
    """The covers of a case, one dict each: w, h, ch, layout, k, plane, header, msg (bytes)."""
    kind = case["kind"]
    if kind == "still":
        one = [dict(w=case["w"], h=case["h"], ch=case["ch"], layout=case["layout"], k=case["k"],
                    plane=case["plane"], header=case["header"], fill=case["fill"])]
    elif kind == "video":
        paper = case["layout"] == "paper"
        one = [dict(w=case["w"], h=case["h"], ch=3, layout=case["layout"], k=1, plane=0 if paper else -1,
                    header=not paper, fill=case["fill"])] * case["frames"]
    else:
        r = random.Random(case["mix"])
        one = []
        for _ in range(case["count"]):
            w, h = _log(r, case["lo"], case["hi"]), _log(r, case["lo"], case["hi"])
            ch = 1 if r.random() < 0.5 else 3
            fill, plane = r.uniform(0.05, 1.0), r.randrange(ch)
            layout = case.get("layout", "stream")
            one.append(dict(w=w, h=h, ch=ch, layout=layout, k=1, plane=plane if layout == "paper" else -1,
                            header=layout == "stream", fill=fill))
    for c in one:
        c["bytes"] = c["w"] * c["h"] * c["ch"]
        if c["layout"] == "paper":
            cap = c["w"] // 4 * c["h"]
        else:
            carry = c["bytes"] if c["plane"] < 0 else c["w"] * c["h"]
            cap = max(0, carry * c["k"] // 8 - (HEADER_BYTES if c["header"] else 0))
        c["msg"] = int(cap * c["fill"])
    return one


def _carrying(c):
    """Bytes of the image that hold the stream, and the bytes that memory has to deliver for them: the colour
    planes lie within each other's 32-byte sectors, so carrying in one plane moves whole pixels."""
    if c["layout"] == "paper":
        return 4 * c["msg"] * c["ch"]
    n = -(-8 * (c["msg"] + (HEADER_BYTES if c["header"] else 0)) // c["k"])
    return min(c["bytes"], n * (c["ch"] if c["plane"] >= 0 else 1))


def work(case):
    total = 0
    for i, c in enumerate(_covers(case)):
        carry = _carrying(c)
        embed = 2 * (carry if case.get("inplace") else c["bytes"]) + c["msg"]
        extract = carry + c["msg"]
        if case["kind"] == "serve":
            total += extract if _reads(i) else embed
        else:
            total += embed + extract + (2 * c["bytes"] if case.get("quality") else 0)
    return {"bytes": float(total), "flops": 0.0}


def _reads(i):
    """Whether request i of a burst extracts: three of every ten."""
    return i % 10 in (2, 5, 8)


# -- inputs --------------------------------------------------------------------


def _random(n, g):
    return torch.randint(0, 256, (n,), dtype=torch.uint8, device="cuda", generator=g)


def _slots(sizes, align):
    """Where buffers of these sizes start in one arena, each at a multiple of `align`, and the arena's size."""
    at, end = [], 0
    for n in sizes:
        at.append(end)
        end += -(-n // align) * align
    return at, end


def _inputs(case, seed):
    """The covers and messages of a case: two arenas, and where each cover and message starts in them."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    covers = _covers(case)
    if case["kind"] == "still":
        c = covers[0]
        cover = _random(c["bytes"] + case["cover_at"], g)
        return covers, cover, [case["cover_at"]], _random(c["msg"] + case["msg_at"], g), [case["msg_at"]]
    align = {"batch": case.get("align"), "video": 1}.get(case["kind"], 256)
    cover_at, n = _slots([c["bytes"] for c in covers], align)
    msg_at, m = _slots([c["msg"] for c in covers], align)
    cover = _random(n, g)
    if case["kind"] == "video":
        h, w, frames = case["h"], case["w"], case["frames"]
        y = (torch.arange(h, device="cuda") * 239 // (h - 1)).view(h, 1, 1)
        x = (torch.arange(w, device="cuda") * 239 // (w - 1)).view(1, w, 1)
        base = (x + y) // 2 + 7 * torch.arange(3, device="cuda").view(1, 1, 3)
        view = cover.view(frames, h, w, 3)
        view &= 15
        for f in range(frames):
            view[f] += ((base + f) % 240).to(torch.uint8)
    return covers, cover, cover_at, _random(max(m, 1), g), msg_at


def _flags(c):
    if c["layout"] == "paper":
        return S.LAYOUT_PAPER2
    return (S.BITS(c["k"]) | (S.HEADER_BE32 if c["header"] else 0) | (S.PLANE_ONLY if c["plane"] >= 0 else 0))


def _records(covers, dtype):
    """Descriptors, requests or jobs of the covers, without their buffers."""
    a = np.zeros(len(covers), dtype=dtype)
    a["cover_bytes"] = [c["bytes"] for c in covers]
    a["msg_bytes"] = a["msg_len"] = [c["msg"] for c in covers]
    a["flags"] = [_flags(c) for c in covers]
    a["width"] = [c["w"] for c in covers]
    a["height"] = [c["h"] for c in covers]
    a["channels"] = [c["ch"] for c in covers]
    a["plane"] = [max(c["plane"], 0) for c in covers]
    return a


def _address(t, at):
    return np.uint64(t.data_ptr()) + np.asarray(at, dtype=np.uint64)


def prepare(case, seed):
    covers, cover, cover_at, msg, msg_at = _inputs(case, seed)
    st = {"kind": case["kind"], "case": case, "n": len(covers)}
    if case["kind"] == "still":
        c = covers[0]
        a, b = case["cover_at"], case["stego_at"]
        st["cover"] = cover[a:]
        st["stego"] = st["cover"] if case["inplace"] else torch.zeros(c["bytes"] + b, dtype=torch.uint8, device="cuda")[b:]
        st["msg"] = msg[case["msg_at"]:]
        st["out"] = torch.zeros_like(msg)[case["msg_at"]:]
        st["geom"] = S.Geom(c["w"], c["h"], c["ch"], max(c["plane"], 0))
        st["flags"], st["len"] = _flags(c), c["msg"]
        st["res"], st["res_x"], st["diff"] = S.new_result(), S.new_result(), torch.zeros(2, dtype=torch.int64, device="cuda")
        return st
    n = len(covers)
    if case["kind"] == "host":
        host = lambda t: torch.empty(t.numel(), dtype=torch.uint8, pin_memory=True).copy_(t)  # noqa: E731
        cover, msg = host(cover), host(msg)
        blank = lambda t: torch.zeros(t.numel(), dtype=torch.uint8, pin_memory=True)  # noqa: E731
        stego, out, again = blank(cover), blank(msg), blank(msg)
        jobs = _records(covers, S.HOST_JOB_DTYPE)
        jobs["cover"], jobs["stego"], jobs["msg"] = _address(cover, cover_at), _address(stego, cover_at), _address(msg, msg_at)
        back = jobs.copy()
        back["cover"], back["msg"], back["stego"] = jobs["stego"], _address(out, msg_at), 0
        jobs["readback"] = _address(again, msg_at)
        st.update(pipe=S.Pipeline(slots=3), jobs=jobs, back=back, keep=(cover, msg), stego=stego, out=out, again=again)
        return st
    stego, out = torch.zeros_like(cover), torch.zeros_like(msg)
    st.update(stego=stego, out=out, keep=(cover, msg))
    if case["kind"] == "serve":
        reads = [i for i in range(n) if _reads(i)]
        if reads:  # what the reading requests read: stegos made beforehand
            d = _records([covers[i] for i in reads], S.DESC_DTYPE)
            for key, t, at in (("cover", cover, cover_at), ("stego", stego, cover_at), ("msg", msg, msg_at)):
                d[key] = _address(t, at)[reads]
            ws = torch.empty(S.stego_batched_workspace_bytes(len(reads)), dtype=torch.uint8, device="cuda")
            S.stego_embed_batched(S.descs_to_device(d), len(reads), S.new_result(n=len(reads)), 0, ws)
            torch.cuda.synchronize()
        r = _records(covers, S.REQUEST_DTYPE)
        is_read = np.array([_reads(i) for i in range(n)])
        r["op"] = np.where(is_read, S.OP_EXTRACT, S.OP_EMBED)
        r["cover"] = np.where(is_read, _address(stego, cover_at), _address(cover, cover_at))
        r["stego"] = np.where(is_read, 0, _address(stego, cover_at))
        r["msg"] = np.where(is_read, _address(out, msg_at), _address(msg, msg_at))
        r["tag"] = np.arange(n)
        st.update(server=S.Server(slots=8, max_batch=512), requests=r)
        return st
    d = _records(covers, S.DESC_DTYPE)
    d["cover"], d["stego"], d["msg"] = _address(cover, cover_at), _address(stego, cover_at), _address(msg, msg_at)
    x = d.copy()
    x["cover"], x["msg"], x["stego"] = d["stego"], _address(out, msg_at), 0
    st["descs"], st["descs_x"] = S.descs_to_device(d), S.descs_to_device(x)
    st["res"], st["res_x"] = S.new_result(n=n), S.new_result(n=n)
    st["ws"] = torch.empty(S.stego_batched_workspace_bytes(n), dtype=torch.uint8, device="cuda")
    if case["kind"] == "video":
        torch.cuda.synchronize()
        st["graph"] = S.BatchedGraph(S.OP_EMBED_BATCHED, st["descs"], n, st["res"], S.FUSE_STATS, st["ws"])
        st["graph_x"] = S.BatchedGraph(S.OP_EXTRACT_BATCHED, st["descs_x"], n, st["res_x"], 0, st["ws"])
    return st


# -- one pass ------------------------------------------------------------------


def run(st):
    kind, n = st["kind"], st["n"]
    if kind == "still":
        flags, geom = st["flags"], st["geom"]
        stats = S.FUSE_STATS if st["case"]["stats"] else 0
        S.stego_embed(st["cover"], st["stego"], st["msg"], flags | stats, st["res"], geom)
        if st["case"]["quality"]:
            S.stego_changed_bytes(st["cover"], st["stego"], st["diff"])
        S.stego_extract(st["stego"], st["out"], st["len"], flags, st["res_x"], geom)
        return {"stego": st["stego"], "message": st["out"], "embedded": st["res"], "extracted": st["res_x"],
                "difference": st["diff"]}
    if kind == "serve":
        st["server"].submit(st["requests"])
        st["server"].drain()
        done = st["server"].poll(n)
        done = done[np.argsort(done["tag"])]
        return {"stego": st["stego"], "message": st["out"],
                "done": [done[key].astype(np.int64) for key in ("tag", "changed", "sse", "msg_bytes", "status")]}
    if kind == "host":
        res, seen = st["pipe"].embed(st["jobs"], S.FUSE_STATS, readback_results=True, raw=True)
        res_x = st["pipe"].extract(st["back"], raw=True)
        return {"stego": st["stego"], "message": st["out"], "checked": st["again"], "embedded": res,
                "seen": seen, "extracted": res_x}
    if kind == "video":
        st["graph"].launch()
        st["graph_x"].launch()
    else:
        S.stego_embed_batched(st["descs"], n, st["res"], S.FUSE_STATS, st["ws"])
        S.stego_extract_batched(st["descs_x"], n, st["res_x"], 0, st["ws"])
    return {"stego": st["stego"], "message": st["out"], "embedded": st["res"], "extracted": st["res_x"]}


# -- the same results in plain torch -------------------------------------------


def _hide(cover, msg, c):
    """The stego of one cover, straight from the layout's definition."""
    dev = cover.device
    stego = cover.clone()
    if c["layout"] == "paper":
        q = c["w"] // 4
        o = torch.arange(c["msg"], device=dev)
        row, j = o // q, o % q
        length = torch.clamp(c["msg"] - row * q, max=q)  # message bytes of that row
        for i in range(4):
            at = (row * c["w"] + length * i + j) * c["ch"] + c["plane"]
            stego[at] = (cover[at] & 0xFC) | ((msg >> (2 * i)) & 3)
        return stego
    s = msg
    if c["header"]:
        head = torch.tensor(list((8 * c["msg"]).to_bytes(4, "big")), dtype=torch.uint8, device=dev)
        s = torch.cat([head, msg])
    k, ch = c["k"], c["ch"] if c["plane"] >= 0 else 1
    bits = (s.view(-1, 1) >> torch.arange(7, -1, -1, dtype=torch.uint8, device=dev)).view(-1) & 1
    n = -(-bits.numel() // k)
    lines = stego[max(c["plane"], 0)::ch]
    old = lines[:n].clone()
    pad = n * k - bits.numel()
    keep = torch.zeros(n, dtype=torch.uint8, device=dev)
    new = torch.zeros(n, dtype=torch.uint8, device=dev)
    full = torch.cat([bits, torch.zeros(pad, dtype=torch.uint8, device=dev)]).view(n, k)
    used = torch.cat([torch.ones_like(bits), torch.zeros(pad, dtype=torch.uint8, device=dev)]).view(n, k)
    for b in range(k):
        keep |= used[:, b] << (k - 1 - b)
        new |= full[:, b] << (k - 1 - b)
    lines[:n] = (old & ~keep) | new
    return stego


def exact(case, seed):
    if case["kind"] not in ("still", "batch") or work(case)["bytes"] > 4e9:
        return None
    covers, cover, cover_at, msg, msg_at = _inputs(case, seed)
    stego, out = torch.zeros_like(cover), torch.zeros_like(msg)
    res, res_x, diff = [], [], torch.zeros(2, dtype=torch.int64, device="cuda")
    for c, a, m in zip(covers, cover_at, msg_at):
        text = msg[m:m + c["msg"]]
        old = cover[a:a + c["bytes"]]
        new = _hide(old, text, c)
        stego[a:a + c["bytes"]] = new
        out[m:m + c["msg"]] = text
        d = new.to(torch.int16) - old.to(torch.int16)
        moved = [int((d != 0).sum()), int((d.to(torch.int32) ** 2).sum())]
        res.append((moved if case.get("stats", True) else [0, 0]) + [c["msg"], 0])
        res_x.append([0, 0, c["msg"], 0])
        if case.get("quality"):
            diff = torch.tensor(moved, dtype=torch.int64)
    if case["kind"] == "still":
        return {"stego": stego[case["cover_at"]:], "message": out[case["msg_at"]:], "embedded": torch.tensor(res[0]),
                "extracted": torch.tensor(res_x[0]), "difference": diff}
    return {"stego": stego, "message": out, "embedded": torch.tensor(res), "extracted": torch.tensor(res_x)}
