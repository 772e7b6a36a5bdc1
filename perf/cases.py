"""What is timed: calls of the package's public entry points as a program that filters streams makes them.

Kinds of case (the "kind" of a case dict):

  stream  a whole stream, or a long piece of one, in one push: the handle is reset, the frames are pushed; with
          "close" the stream is then closed (candidates) and its candidate frames, as many as the encoder's batch
          holds, are gathered into that batch's buffer
  live    the next frames of a running stream, pushed as they arrive, into output buffers that the program keeps
  graph   a stream's pushes captured once into a CUDA graph, launched again for the next frames in the same buffers
  serve   one batched call for many streams with a few new frames each, descriptors laid out once per buffer slot
  qer     one query: candidate frames ranked by text-to-vision attention, the best kept

Frames are seeded scenes: a smooth random texture per scene, moved by a few pixels and with a slow change of
brightness from frame to frame, and noise; scene lengths are geometric. Queries and keys are bf16 Gaussian draws, with
the keys of a few frames leaning towards one text token. With "features" the program also takes each frame's
features (of the hash signal, the hashes that it keeps).
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2609_03675_gb300 import NGFF, QER

HISTOGRAM, LOWRES, DHASH, SCD = 0, 1, 2, 3
LUMA = (299, 587, 114, 1000)


def _stream(name, width, height, n, **kw):
    c = {"name": name, "kind": "stream", "width": width, "height": height, "n": n, "bins": 32, "l_max": 30, "tau": 0.30,
         "signal": HISTOGRAM, "features": False, "close": False, "scene": 40}
    c.update(kw)
    return c


def _qer(name, n_text, frames, tokens, **kw):
    c = {"name": name, "kind": "qer", "n_text": n_text, "frames": frames, "tokens": tokens, "heads": 32, "kv_heads": 8,
         "head_dim": 128, "rho": 0.3, "wait": False}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: a live camera, one 1080p frame at a time
        {"name": "live_1080p", "kind": "live", "width": 1920, "height": 1080, "n": 1, "pool": 48, "bins": 32, "l_max": 30,
         "tau": 0.30, "signal": HISTOGRAM, "features": False, "scene": 20},
        # a short clip at the encoder's own size, pushed all at once
        _stream("clip_224", 224, 224, 64, scene=16),
        # ten minutes at 1 frame/s in pushes of 8, launched from one CUDA graph
        {"name": "chunks_448", "kind": "graph", "width": 448, "height": 448, "n": 8, "pushes": 75, "bins": 32, "l_max": 30,
         "tau": 0.30, "signal": HISTOGRAM, "features": False, "scene": 20},
        # a server: 32 streams of 640x360 with 1 to 8 new frames each per call
        {"name": "serve_32x360p", "kind": "serve", "width": 640, "height": 360, "streams": 32, "most": 8, "slots": 6,
         "bins": 32, "l_max": 30, "tau": 0.30, "signal": HISTOGRAM, "scene": 20},
        # the largest: a whole 1080p stream pushed, closed, and its candidates gathered
        _stream("stream_1080p", 1920, 1080, 1200, close=True, scene=150),
        # the low-resolution copy of a long stream: many small frames, where the selection shows beside the histograms
        _stream("long_224", 224, 224, 4096, scene=20),
        # no forced retention, with scene changes
        _stream("scenes_nogap_360p", 640, 360, 2048, l_max=0, tau=0.15, signal=SCD, scene=20),
        # full-resolution histograms and a long retention interval
        _stream("bins256_720p", 1280, 720, 480, bins=256, l_max=60, tau=0.15, scene=60),
        # the block-difference signal on 480p video, whose width is no multiple of 16
        _stream("lowres_854x480", 854, 480, 600, signal=LOWRES, tau=0.05, scene=40),
        # frames whose size no vector width divides, closed and gathered
        _stream("odd_1917x1080", 1917, 1080, 300, close=True, scene=40),
        # a query over a long prefix: 1024 candidates of 256 tokens, 256 text tokens
        _qer("query_1024", 256, 1024, 256),
        # an interactive query: a short question over 32 candidates, its answer awaited
        _qer("query_32_short", 40, 32, 256, wait=True),
    ]


SIZES = ((224, 224), (336, 336), (448, 448), (426, 240), (640, 360), (854, 480), (960, 540), (1280, 720), (1366, 768),
         (1920, 1080), (1080, 1920), (2560, 1440), (3840, 2160), (1917, 1080), (641, 359), (333, 251), (97, 113))


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("stream", "stream", "stream", "live", "graph", "serve", "qer", "qer"))
    if kind == "qer":
        heads, kv_heads, head_dim = rng.choice(((32, 8, 128), (32, 8, 128), (28, 4, 128), (16, 8, 64), (16, 16, 64), (14, 2, 64)))
        tokens = rng.choice((49, 64, 100, 144, 196, 256, 256, 400))
        n_text = _log(rng, 8, 1024)
        frames = _log(rng, 4, max(4, min(1024, int(1024 * 256 * 256 / (tokens * max(n_text, 256))))))
        c = _qer("", n_text, frames, tokens, heads=heads, kv_heads=kv_heads, head_dim=head_dim, rho=rng.choice((0.1, 0.3, 0.5)),
                 wait=rng.random() < 0.5)
        del c["name"]
        return c
    if rng.random() < 0.6:
        width, height = rng.choice(SIZES)
    else:
        width, height = _log(rng, 64, 2000), _log(rng, 64, 1200)
    frame = 3 * width * height
    signal = rng.choice((HISTOGRAM, HISTOGRAM, HISTOGRAM, HISTOGRAM, LOWRES, DHASH, SCD))
    if kind == "serve" and signal == DHASH:  # a batched call hands out no features
        signal = LOWRES
    spatial = signal in (LOWRES, DHASH)
    c = {"kind": kind, "width": width, "height": height, "bins": 32 if spatial else rng.choice((16, 32, 32, 32, 48, 64, 128, 256)),
         "l_max": rng.choice((0, 15, 30, 30, 30, 45, 120)), "tau": rng.choice((0.05, 0.1)) if spatial else rng.choice((0.1, 0.15, 0.3)),
         "signal": signal, "scene": rng.choice((10, 20, 60, 150))}
    if kind != "serve":
        c["features"] = signal == DHASH or rng.random() < 0.1
    if kind == "stream":
        c["n"] = _log(rng, 16, max(16, min(4096, int(2.0e9 / frame))))
        c["close"] = rng.random() < 0.4
    elif kind == "live":
        c["n"] = rng.choice((1, 1, 2, 4, 8, 16))
        c["pool"] = c["n"] * max(2, min(64, int(4.0e8 / (frame * c["n"]))))
    elif kind == "graph":
        c["n"] = rng.choice((1, 2, 4, 8, 16, 48))
        c["pushes"] = max(2, min(75, int(6.0e8 / (frame * c["n"]))))
    else:
        c["streams"] = max(2, min(rng.choice((4, 8, 16, 32, 64)), int(2.5e8 / (4.5 * frame))))
        c["most"] = rng.choice((1, 4, 8))
        c["slots"] = 4
    return c


# ---------------------------------------------------------------------- inputs


def _scenes(n, width, height, seed, mean):
    """n seeded frames, uint8 [n, height, width, 3] on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = random.Random(seed)
    pad = 16
    frames = torch.empty((n, height, width, 3), dtype=torch.uint8, device="cuda")
    noise = torch.randint(-3, 4, (height + pad, width + pad, 3), generator=g, device="cuda", dtype=torch.int16)
    noise += torch.randint(-2, 3, noise.shape, generator=g, device="cuda", dtype=torch.int16)
    value = torch.empty((height, width, 3), dtype=torch.int16, device="cuda")
    t = 0
    while t < n:
        length = 1
        while r.random() > 1.0 / mean:
            length += 1
        tex = torch.zeros((1, 3, height + pad, width + pad), device="cuda")
        for cells, weight in ((4, 0.7), (24, 0.3)):
            grid = torch.rand((1, 3, cells, cells), generator=g, device="cuda")
            tex += weight * torch.nn.functional.interpolate(grid, size=tex.shape[2:], mode="bilinear")
        base = (r.uniform(20.0, 110.0) + r.uniform(50.0, 150.0) * tex)[0].permute(1, 2, 0).to(torch.int16).contiguous()
        y = x = pad // 2
        light, step = 0, r.choice((-1, 0, 0, 1))
        for _ in range(min(length, n - t)):
            y, x = min(pad, max(0, y + r.randint(-2, 2))), min(pad, max(0, x + r.randint(-2, 2)))
            light = max(-40, min(40, light + step))
            ny, nx = r.randint(0, pad), r.randint(0, pad)
            torch.add(base[y:y + height, x:x + width], noise[ny:ny + height, nx:nx + width], out=value)
            value.add_(light).clamp_(0, 255)
            frames[t].copy_(value)
            t += 1
    return frames


def _handle(case, streams=1):
    return NGFF(case["width"], case["height"], bins=case["bins"], l_max=case["l_max"], tau=case["tau"], signal=case["signal"],
                max_streams=streams)


def _new_frames(case):
    """The frames that each stream gets in each call of a "serve" case: counts[slot][stream]."""
    r = random.Random(case["streams"])
    return [[r.randint(1, case["most"]) for _ in range(case["streams"])] for _ in range(case["slots"])]


def _query(case, seed):
    """q [n_text, heads, head_dim] and k [frames * tokens, kv_heads, head_dim], bf16 on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = random.Random(seed)
    d, kv = case["head_dim"], case["kv_heads"]
    q = torch.randn((case["n_text"], case["heads"], d), generator=g, device="cuda")
    k = torch.randn((case["frames"] * case["tokens"], kv, d), generator=g, device="cuda")
    for f in r.sample(range(case["frames"]), min(8, case["frames"])):
        lean = q[r.randrange(case["n_text"])].view(kv, case["heads"] // kv, d).mean(dim=1)
        lean = lean / lean.norm(dim=-1, keepdim=True) * (1.5 * math.sqrt(d) / 4)
        k[f * case["tokens"]:(f + 1) * case["tokens"]] += lean
    return q.to(torch.bfloat16), k.to(torch.bfloat16)


def _kept(case):
    return max(1, round(float(np.float32(case["rho"])) * case["frames"]))


def _batch(case):
    """Frames that the encoder's batch holds."""
    return 16 + case["n"] // 16


def _before(case):
    """Frames of a "live" case's pool that are pushed before the first pass."""
    return case["pool"] // (2 * case["n"]) * case["n"]


def _outputs(f, n, features=False):
    out = {"scores": torch.empty(n, dtype=torch.float32, device="cuda"), "keep": torch.empty(n, dtype=torch.uint8, device="cuda")}
    if features:
        out["hist"] = torch.empty((n, f.feature_words), dtype=torch.int32, device="cuda")
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "qer":
        q, k = _query(case, seed)
        f = QER(case["n_text"], case["heads"], case["kv_heads"], case["head_dim"], case["frames"], case["tokens"], case["rho"])
        return {"case": case, "qer": f, "q": q, "k": k, "w": torch.empty(case["frames"], dtype=torch.float32, device="cuda"),
                "sel": torch.zeros(case["frames"], dtype=torch.int32, device="cuda"),
                "count": torch.zeros(1, dtype=torch.int32, device="cuda"), "kept": _kept(case)}
    size = (case["width"], case["height"])
    if kind == "stream":
        state = {"case": case, "ngff": _handle(case), "frames": _scenes(case["n"], *size, seed, case["scene"])}
        if case["close"]:
            state["batch"] = torch.zeros((_batch(case), size[1], size[0], 3), dtype=torch.uint8, device="cuda")
        return state
    if kind == "live":  # a stream that has been running for a while: the first half of the pool has been pushed
        frames = _scenes(case["pool"], *size, seed, case["scene"])
        f = _handle(case)
        f.push(frames[:_before(case)])
        return {"case": case, "ngff": f, "frames": frames, "out": _outputs(f, case["n"], case["features"]), "at": _before(case)}
    if kind == "graph":
        n = case["n"] * case["pushes"]
        frames = _scenes(n, *size, seed, case["scene"])
        f = _handle(case)
        out = _outputs(f, n, case["features"])
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            for i in range(0, n, case["n"]):
                j = i + case["n"]
                f.push(frames[i:j], **{name: out[name][i:j] for name in out})
        return {"case": case, "ngff": f, "frames": frames, "out": out, "graph": graph}
    f = _handle(case, case["streams"])
    slots = []
    for s, counts in enumerate(_new_frames(case)):  # the buffers that the decoders fill, and their descriptors
        frames = _scenes(sum(counts), *size, seed * 64 + s, case["scene"])
        out = _outputs(f, sum(counts))
        items, at = [], 0
        for stream, n in enumerate(counts):
            items.append((stream, frames[at:at + n], out["scores"][at:at + n], out["keep"][at:at + n]))
            at += n
        slots.append({"frames": frames, "out": out, "batch": f.make_batch(items)})
    return {"case": case, "ngff": f, "slots": slots, "at": 0}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "qer":
        if case["wait"]:
            w, sel = state["qer"].run(state["q"], state["k"])
        else:
            state["qer"].run_async(state["q"], state["k"], state["w"], state["sel"], state["count"])
            w, sel = state["w"], state["sel"][: state["kept"]]
        return {"scores": w, "selected": sel}
    f = state["ngff"]
    if kind == "stream":
        f.reset()
        out = dict(zip(("scores", "keep", "hist"), f.push(state["frames"], return_hist=case["features"])))
        if case["close"]:
            idx = f.candidates()
            taken = idx[: _batch(case)]
            f.gather(state["frames"], taken, out=state["batch"][: taken.numel()])
            out.update(candidates=idx.numel(), batch=state["batch"])
        return out
    if kind == "live":
        at = state["at"]
        state["at"] = (at + case["n"]) % case["pool"]
        f.push(state["frames"][at:at + case["n"]], **state["out"])
        return state["out"]
    if kind == "graph":
        state["graph"].replay()
        return state["out"]
    slot = state["slots"][state["at"]]
    state["at"] = (state["at"] + 1) % len(state["slots"])
    f.push_batch_raw(*slot["batch"])
    return slot["out"]


def _frames_of(case):
    """Frames of one pass, and the frames that closing them hands on at least."""
    kind = case["kind"]
    if kind == "graph":
        return case["n"] * case["pushes"], 0
    if kind == "serve":
        return sum(map(sum, _new_frames(case))) / case["slots"], 0
    if kind == "stream" and case["close"]:
        return case["n"], min(_batch(case), 1 + case["n"] // (case["l_max"] or case["scene"]))
    return case["n"], 0


def work(case):
    if case["kind"] == "qer":
        D, nv = case["kv_heads"] * case["head_dim"], case["frames"] * case["tokens"]
        return {"bytes": 2 * nv * D + 2 * case["n_text"] * case["heads"] * case["head_dim"] + 4 * case["frames"] + 4 * _kept(case),
                "flops": 2 * case["n_text"] * nv * D}
    n, kept = _frames_of(case)
    frame = 3 * case["width"] * case["height"]
    words = {LOWRES: 256, DHASH: 2}.get(case["signal"], case["bins"]) if case.get("features") else 0
    return {"bytes": n * (frame + 5 + 4 * words) + 2 * kept * frame, "flops": 0}


def tolerance(case):
    if case["kind"] == "qer":
        # sums of up to 1024 bf16 products in fp32, in another order; a near tie at the cut may fall either way
        return {"rel": 4e-6, "max": 2e-5, "differ": 0.01}
    # integer counts, then one fp32 division: keep codes, indices and frames are exact
    return {"rel": 2.5e-7, "max": 1e-6, "differ": 0.0}


# ----------------------------------------------------------- 64-bit references


def _luma(frames):
    x = frames.to(torch.int64)
    wr, wg, wb, den = LUMA
    return (x[..., 0] * wr + x[..., 1] * wg + x[..., 2] * wb + den // 2) // den


def _features(case, frames):
    """One row of whole numbers per frame: counts, cell sums or hash bits (numpy int64)."""
    H, W, rows = case["height"], case["width"], []
    per = max(1, int(4.0e7 / (H * W)))
    grid = {LOWRES: (16, 16), DHASH: (8, 9)}.get(case["signal"])
    if grid:
        gh, gw = grid
        cy, cx = torch.arange(H, device="cuda") * gh // H, torch.arange(W, device="cuda") * gw // W
        R = torch.nn.functional.one_hot(cy, gh).double().T.contiguous()
        C = torch.nn.functional.one_hot(cx, gw).double()
        count = R.sum(1)[:, None] * C.sum(0)[None, :]
    for i in range(0, frames.shape[0], per):
        y = _luma(frames[i:i + per])
        m = y.shape[0]
        if grid:
            S = R @ y.double() @ C
            if case["signal"] == DHASH:
                S = (S[:, :, :-1] * count[:, 1:] > S[:, :, 1:] * count[:, :-1])
            rows.append(S.reshape(m, -1).to(torch.int64).cpu().numpy())
        else:
            at = (y * case["bins"] // 256 + torch.arange(m, device="cuda")[:, None, None] * case["bins"]).reshape(-1)
            rows.append(torch.bincount(at, minlength=m * case["bins"]).view(m, -1).cpu().numpy())
    return np.concatenate(rows)


def _rule(case, feat):
    """(scores in 64 bits, keep codes) of a stream from its first frame; decisions in 32 bits, as the rule defines them."""
    N = case["width"] * case["height"]
    den = {LOWRES: 255 * N, DHASH: 64}.get(case["signal"], 2 * N)
    reaches = lambda x, thr: np.float32(x) / np.float32(den) >= np.float32(thr)  # noqa: E731
    scores, keep = np.zeros(len(feat)), np.zeros(len(feat), dtype=np.int64)
    adj = np.abs(np.diff(feat, axis=0)).sum(axis=1)
    last, run = 0, 0
    keep[0] = 3
    for t in range(1, len(feat)):
        a = int(adj[t - 1])
        x = max(a, int(np.abs(feat[t] - feat[last]).sum()))
        scores[t] = x / den
        scene = False
        if case["signal"] == SCD:
            if reaches(a, 0.30):
                scene, run = True, 0
            elif reaches(a, 0.10):
                run += a
                scene = reaches(run, 0.30) and not reaches(run - a, 0.30)
            else:
                run = 0
        if reaches(x, case["tau"]):
            keep[t] = 1
        elif scene:
            keep[t] = 4
        elif case["l_max"] and t - last >= case["l_max"]:
            keep[t] = 2
        if keep[t]:
            last = t
    return scores, keep


def exact(case, seed):
    kind = case["kind"]
    if kind == "qer":
        q, k = _query(case, seed)
        n, d, kv = case["n_text"], case["head_dim"], case["kv_heads"]
        q = q.double().view(n, kv, case["heads"] // kv, d).sum(dim=2).reshape(n, kv * d)
        best = torch.cat([(k[i:i + 32768].double().reshape(-1, kv * d) @ q.T).amax(dim=1) for i in range(0, k.shape[0], 32768)])
        w = best.view(case["frames"], case["tokens"]).mean(dim=1) / (case["heads"] * math.sqrt(d))
        order = torch.argsort(w, descending=True, stable=True)[:_kept(case)]
        return {"scores": w, "selected": torch.sort(order).values}
    size = (case["width"], case["height"])
    if kind == "serve":
        counts = _new_frames(case)[0]
        feat = _features(case, _scenes(sum(counts), *size, seed * 64, case["scene"]))
        parts = [_rule(case, part) for part in np.split(feat, np.cumsum(counts)[:-1])]
        return {"scores": np.concatenate([p[0] for p in parts]), "keep": np.concatenate([p[1] for p in parts])}
    first = _before(case) if kind == "live" else 0
    n = first + case["n"] * case.get("pushes", 1)
    scores, keep = _rule(case, _features(case, _scenes(n, *size, seed, case["scene"])))
    return {"scores": scores[first:], "keep": keep[first:], "hist": None, "candidates": None, "batch": None}
