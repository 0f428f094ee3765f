"""The work a program has this framework do, as measurable cases.

Each case is one pass through the public entry points: a search of a cube of
dirty images (device cube in, candidate list or FULL arrays out), the longer
timescales, a serving block, an imaging call, a training step of the candidate
classifier, and the classification of a candidate list.  Sizes come from the
repository's configurations and benchmark (64 x 64 and 301 x 301 fields of 25
samples, 301 x 301 and 512 x 512 windows of 1200 samples, 25-sample serving
blocks, 82-antenna imaging blocks of 175 x 175 pixels, 32^3 x 16 cutouts).

``exact`` restates every result in 64 bits with torch and numpy alone.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2510_18136_gb300 import multiscale, native, synth, synth_vis

DEV = "cuda"
FIELDS = ("row", "col", "dm_idx", "w_idx", "t_idx")
EPS = 0.03          # BF16/FP16 S/N error bound with known noise: the re-score band
C_LIGHT = 299792458.0


def listed():
    return [
        # the smallest call: one small field's 25-sample block (3.35 s), where launches and latency count
        dict(name="block_64", kind="search", ny=64, nx=64, n_sub=16, n_t=25, n_dm=16, dm_max=2000.0, w_max=16,
             dtype="f32", noise="known", out="candidates", rescore=False, threshold=6.0),
        # the real-time block of a whole field: 301 x 301 pixels, 25 samples, 16 DM trials, 5 widths
        dict(name="block_301", kind="search", ny=301, nx=301, n_sub=16, n_t=25, n_dm=16, dm_max=2000.0, w_max=16,
             dtype="f32", noise="known", out="candidates", rescore=False, threshold=6.0),
        # the full 160.8 s window of a field in FP32: the flagship search
        dict(name="window_301_f32", kind="search", ny=301, nx=301, n_sub=16, n_t=1200, n_dm=64, dm_max=2000.0,
             w_max=1200, dtype="f32", noise="known", out="candidates", rescore=False, threshold=6.0),
        # the same window stored in BF16, candidates near the threshold searched again in FP32
        dict(name="window_301_bf16", kind="search", ny=301, nx=301, n_sub=16, n_t=1200, n_dm=64, dm_max=2000.0,
             w_max=1200, dtype="bf16", noise="known", out="candidates", rescore=True, threshold=6.0),
        # a 512 x 512 field of unknown, heavy-tailed noise: MAD normalisation, 256 DM trials, and the
        # real-time threshold of 8.5
        dict(name="mad_512_bf16", kind="search", ny=512, nx=512, n_sub=16, n_t=1200, n_dm=256, dm_max=4000.0,
             w_max=1200, dtype="bf16", noise="mad", out="candidates", rescore=False, threshold=8.5),
        # S/N and arrival time of every (pixel, DM, width), kept on the device (post-processing of a field)
        dict(name="full_arrays_129", kind="search", ny=129, nx=129, n_sub=16, n_t=1200, n_dm=64, dm_max=2000.0,
             w_max=1200, dtype="f32", noise="known", out="full", rescore=False, threshold=6.0),
        # an offline window past the paper's: 2048 samples (275 s)
        dict(name="long_193_2048", kind="search", ny=193, nx=193, n_sub=16, n_t=2048, n_dm=64, dm_max=2000.0,
             w_max=2048, dtype="f32", noise="known", out="candidates", rescore=False, threshold=6.0),
        # the 0.67 s and 10.05 s searches of the full window: binning by 5 and by 75, then their searches
        dict(name="timescales_301", kind="timescales", ny=301, nx=301, n_sub=16, n_t=1200, n_dm=64, dm_max=2000.0,
             dtype="f32", threshold=6.0),
        # one 25-sample block of a served 301 x 301 field (BF16 window of 1200 samples, re-scoring on)
        dict(name="serve_301", kind="serve", ny=301, nx=301, n_sub=16, n_t=1200, n_dm=64, dm_max=2000.0, w_max=1200,
             n_blk=25, dtype="bf16", threshold=6.0),
        # dirty images of one 25-sample block: 16 subbands x 8 channels x 3321 baselines -> 400 images of 175 x 175
        dict(name="image_block", kind="image", n_t=25, n_sub=16, n_chan=8, n_ew=48, n_ns=34, n_grid=175),
        # one training step of the candidate classifier, batch 64 (forward, backward, Adam)
        dict(name="train_64", kind="train", batch=64, d=32, hw=32, c0=16, chans="32-32-64-64", f=32, dropout=0.5),
        # a search's candidates through the classifier: cutouts from the cube, then inference
        dict(name="classify_256", kind="classify", ny=128, nx=128, n_sub=16, n_t=256, n_dm=64, dm_max=2000.0,
             w_max=128, n_cand=256, d=32, hw=32, chans="32-32-64-64", f=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search"] * 6 + ["timescales", "serve", "image", "train", "classify"])
    if kind == "image":
        return dict(kind="image", n_t=_log(rng, 1, 40), n_sub=rng.choice([4, 8, 16]), n_chan=rng.randint(1, 8),
                    n_ew=rng.randint(12, 48), n_ns=rng.randint(8, 34), n_grid=rng.randint(64, 257))
    if kind == "train":
        return dict(kind="train", batch=_log(rng, 4, 96), d=rng.choice([16, 32]), hw=rng.choice([16, 32, 32]),
                    c0=rng.choice([8, 16]), chans=rng.choice(["32-32-64-64", "16-32-32-64", "32-64-64-64"]),
                    f=rng.choice([16, 32, 64]), dropout=rng.choice([0.0, 0.25, 0.5]))
    if kind == "classify":
        return dict(kind="classify", ny=rng.randint(48, 160), nx=rng.randint(48, 160), n_sub=16,
                    n_t=rng.randint(100, 400), n_dm=_log(rng, 8, 64), dm_max=rng.uniform(1000.0, 4000.0), w_max=64,
                    n_cand=_log(rng, 1, 300), d=rng.choice([16, 32]), hw=rng.choice([16, 32]),
                    chans=rng.choice(["32-32-64-64", "16-32-32-64"]), f=32)
    side = (24, 301)
    c = dict(kind=kind, ny=_log(rng, *side), nx=_log(rng, *side), n_sub=rng.choice([8, 12, 16, 16, 16, 20]),
             n_t=0, n_dm=_log(rng, 4, 128), dm_max=rng.uniform(500.0, 4000.0))
    if kind == "timescales":
        c.update(n_t=rng.randint(300, 1400), dtype=rng.choice(["f32", "bf16", "f16"]), threshold=6.0)
    elif kind == "serve":
        c.update(n_t=rng.randint(400, 1200), n_blk=rng.randint(5, 32), dtype=rng.choice(["f32", "bf16", "bf16"]),
                 threshold=6.0)
        c["w_max"] = c["n_t"]
    else:
        noise = rng.choice(["known", "known", "known", "mad"])
        out = rng.choice(["candidates"] * 4 + ["full"])
        c.update(n_t=_log(rng, 200, 1800) if noise == "mad" else _log(rng, 16, 3000),
                 dtype=rng.choice(["f32", "f32", "bf16", "f16"]), noise=noise, out=out,
                 threshold=8.5 if noise == "mad" else 6.5)
        c["w_max"] = _log(rng, 1, c["n_t"]) if rng.random() < 0.3 else c["n_t"]
        c["rescore"] = c["dtype"] != "f32" and noise == "known" and out == "candidates" and rng.random() < 0.5
        # no dearer than the listed cases: trials, and the FULL arrays' entries
        per_pix = c["n_dm"] * c["n_t"] * len(_widths(c["w_max"]))
        most = min((1.2e10 if c["n_t"] > 1247 else 5e10) / per_pix,
                   1e7 / (c["n_dm"] * len(_widths(c["w_max"]))) if out == "full" else 1e9, 1.1e5)
        while c["ny"] * c["nx"] > most and min(c["ny"], c["nx"]) > 8:
            c["ny"], c["nx"] = max(8, int(c["ny"] * 0.8)), max(8, int(c["nx"] * 0.8))
    return c


# ------------------------------------------------------------------ what the cases are made of

def _widths(w_max):
    """Powers of two up to min(w_max, 1024), and w_max itself."""
    w = [1 << i for i in range(11) if (1 << i) <= w_max]
    return w if w[-1] == w_max else w + [int(w_max)]


def _config(c, n_t=None, factor=1, dm=None, w_max=None):
    n_t = c["n_t"] if n_t is None else n_t
    dm = np.linspace(0.0, c["dm_max"], c["n_dm"]) if dm is None else dm
    return synth.SearchConfig(ny=c["ny"], nx=c["nx"], n_sub=c["n_sub"], n_t=n_t, t_samp_ms=134.2 * factor,
                              freq_mhz=_freqs(c["n_sub"]), dm=dm,
                              widths=np.array(_widths(w_max or c["w_max"]), np.int32), threshold=c["threshold"])


def _freqs(n_sub):
    return 1311.0 + (np.arange(n_sub) + 0.5) * (187.0 / n_sub)


def _delays(dm, n_sub, t_samp_ms=134.2):
    f = _freqs(n_sub) / 1000.0
    return np.floor(4.149 * np.asarray(dm, float)[:, None] * (f ** -2.0 - f[-1] ** -2.0) / t_samp_ms + 0.5).astype(int)


def _bursts(c, seed, n):
    """n bursts on a field: (row, col, dm, width, S/N, u), u placing the start; 3 px apart, 2 from the edge."""
    rng = np.random.default_rng([seed, 11])
    got = []
    for _ in range(50 * n):
        r, q = int(rng.integers(2, c["ny"] - 2)), int(rng.integers(2, c["nx"] - 2))
        if len(got) < n and all(max(abs(r - a[0]), abs(q - a[1])) >= 3 for a in got):
            w_top = max(1, min(c.get("w_max", c["n_t"]), c["n_t"] // 2))
            got.append((r, q, rng.uniform(0, c["dm_max"]), max(1, round(math.exp(rng.uniform(0, math.log(w_top))))),
                        rng.uniform(6.0, 30.0) + (c["threshold"] - 6.0), rng.uniform()))
    return got


def _field(c, seed):
    """A cube [n_pix, n_sub, n_t] FP32 or 16-bit of noise with bursts (PSF-shaped on PSF noise)."""
    cfg = _config(dict(c, w_max=1))
    mad = c.get("noise") == "mad"
    if mad:
        cube = synth.beam_student_noise(cfg, seed, device=DEV, dtype=torch.float32 if c["dtype"] == "f32"
                                        else torch.bfloat16 if c["dtype"] == "bf16" else torch.float16)
        sig = synth.beam_sigma(cfg)
        psf = np.zeros((5, 5))
        psf[2, 2] = 1.0
    else:
        cube = synth.psf_noise(cfg, seed, device=DEV)
        sig = np.full(cfg.n_pix, synth.psf_sigma())
        psf = synth.gaussian_psf()
    x = cube.view(c["ny"], c["nx"], c["n_sub"], c["n_t"])
    tap = torch.tensor(psf, dtype=torch.float32, device=DEV)[:, :, None]
    for r, q, dm, w, snr, u in _bursts(c, seed, max(3, min(50, cfg.n_pix // 1800))):
        sh = _delays([dm], c["n_sub"])[0]
        w = max(1, min(w, c["n_t"] - sh[0]))
        t0 = int(u * max(1, c["n_t"] - sh[0] - w + 1))
        amp = snr * sig[r * c["nx"] + q] / math.sqrt(c["n_sub"] * w)
        for k in range(c["n_sub"]):
            a = t0 + int(sh[k])
            if a < c["n_t"]:
                x[r - 2:r + 3, q - 2:q + 3, k, a:a + w] += (amp * tap).to(x.dtype)
    return cube


_STORE = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


def _sigma(c, n_pix):
    return torch.full((n_pix,), synth.psf_sigma() * math.sqrt(c["n_sub"]), device=DEV)


def _search_inputs(c, seed):
    cube = _field(c, seed)
    sigma = None if c.get("noise") == "mad" else _sigma(c, cube.shape[0])
    stored = cube if cube.dtype == _STORE[c["dtype"]] else cube.to(_STORE[c["dtype"]])
    return stored, sigma, cube if c.get("rescore") else None


def _serve_blocks(c, seed):
    """The blocks that fill the window, oldest first: [n_blk, n_sub, ny, nx] unit noise; the last one ends bursts."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    n = -(-c["n_t"] // c["n_blk"])
    bursts = _bursts(dict(c, w_max=c["n_t"] // 2), seed, max(3, c["ny"] * c["nx"] // 1800))
    total = n * c["n_blk"]
    for b in range(n):
        blk = torch.randn((c["n_blk"], c["n_sub"], c["ny"], c["nx"]), generator=g, device=DEV)
        at = b * c["n_blk"]
        for r, q, dm, w, snr, u in bursts:
            sh = _delays([dm], c["n_sub"])[0]
            w = max(1, min(w, c["n_t"] - sh[0]))
            t0 = total - 1 - int(u * c["n_blk"]) - sh[0] - w + 1
            for k in range(c["n_sub"]):
                lo, hi = max(t0 + sh[k] - at, 0), min(t0 + sh[k] + w - at, c["n_blk"])
                if lo < hi:
                    blk[lo:hi, k, r, q] += snr / math.sqrt(c["n_sub"] * w)
        yield blk


def _vis(c, seed):
    uv = synth_vis.baseline_uv(synth_vis.core_layout(0, c["n_ew"], c["n_ns"]))
    chan = synth_vis.channel_freqs(c["n_sub"], c["n_chan"])
    rng = np.random.default_rng([seed, 3])
    far = c["n_grid"] // 3
    src = [(int(rng.integers(-far, far + 1)), int(rng.integers(-far, far + 1)), rng.uniform(0.5, 3.0, (c["n_t"], c["n_sub"])))
           for _ in range(4)]
    return uv, chan, synth_vis.visibilities(uv, chan, c["n_t"], src, noise=1.0, seed=seed, device=DEV)


def _chans(c):
    return tuple(int(v) for v in c["chans"].split("-"))


def _clf_layout(c, c0):
    """(name, shape) of the flat parameter vector, in order."""
    out, cin = [], c0
    for l, co in enumerate(_chans(c)):
        out += [("w%d" % l, (co, 27, cin)), ("g%d" % l, (co,)), ("b%d" % l, (co,))]
        cin = co
    fin = (c["d"] // 16) * (c["hw"] // 16) ** 2 * cin
    return out + [("fw", (c["f"], fin)), ("fb", (c["f"],)), ("ow", (c["f"],)), ("ob", (1,))]


def _clf_params(c, c0, seed):
    rng = np.random.default_rng([seed, 5])
    got = []
    for name, shape in _clf_layout(c, c0):
        n = int(np.prod(shape))
        if name[0] == "g":
            got.append(rng.uniform(0.8, 1.2, n))
        elif name[0] == "b" or name in ("fb", "ob"):
            got.append(rng.normal(0.0, 0.05, n))
        else:
            got.append(rng.normal(0.0, math.sqrt(2.0 / np.prod(shape[1:] if len(shape) > 1 else shape)), n))
        if name[0] == "w":      # the convolutions multiply BF16 weights
            got[-1] = torch.from_numpy(got[-1]).to(torch.bfloat16).double().numpy()
    return np.concatenate(got).astype(np.float32)


def _bn_stats(c, seed):
    rng = np.random.default_rng([seed, 6])
    n = sum(_chans(c))
    return rng.normal(0.0, 0.1, n).astype(np.float32), rng.uniform(1.0, 3.0, n).astype(np.float32)


def _train_batch(c, seed):
    """Cutouts of unit noise, half of them with a dispersed track (label 0), half with a zero-DM step (label 1)."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    x = torch.randn((c["batch"], c["d"], c["hw"], c["hw"], c["c0"]), generator=g, device=DEV)
    labels = (torch.arange(c["batch"], device=DEV) % 2).float()
    mid, z = c["hw"] // 2, c["d"] // 2
    x[1::2, z - 2:z + 2] += 0.7
    for k in range(c["c0"]):
        a = z + (c["c0"] - 1 - k) // 4
        x[0::2, a - 2:a + 1, mid - 1:mid + 2, mid - 1:mid + 2, k] += 2.0
    return x.to(torch.bfloat16), labels


def _clf_cands(c, seed):
    rng = np.random.default_rng([seed, 8])
    out = np.zeros(c["n_cand"], native.CANDIDATE_DTYPE)
    out["row"] = rng.integers(0, c["ny"], c["n_cand"])
    out["col"] = rng.integers(0, c["nx"], c["n_cand"])
    out["dm_idx"] = rng.integers(0, c["n_dm"], c["n_cand"])
    out["w_idx"] = rng.integers(0, len(_widths(c["w_max"])), c["n_cand"])
    out["t_idx"] = rng.integers(0, max(1, c["n_t"] - 40), c["n_cand"])
    out["snr"] = rng.uniform(6.0, 30.0, c["n_cand"])
    return out


def _clf(c, c0, batch, seed, dropout):
    clf = native.Classifier(batch=batch, d=c["d"], h=c["hw"], w=c["hw"], c0=c0, c=_chans(c), f=c["f"],
                            dropout=dropout, seed=7, lr=1e-3)
    clf.set_params(_clf_params(c, c0, seed))
    clf.set_bn_stats(*_bn_stats(c, seed))
    return clf


# ------------------------------------------------------------------ the cases' functions

def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "search":
        cube, sigma, cube32 = _search_inputs(c, seed)
        plan = native.Plan(_config(c), dtype=c["dtype"], noise=c["noise"], out=c["out"],
                           rescore_eps=EPS if c["rescore"] else 0.0)
        s = dict(kind=kind, plan=plan, cube=cube, sigma=sigma, cube32=cube32, full=c["out"] == "full")
        if s["full"]:
            shape = (plan.cfg.n_pix, c["n_dm"], len(plan.cfg.widths))
            s["snr"] = torch.empty(shape, dtype=torch.float32, device=DEV)
            s["toa"] = torch.empty(shape, dtype=torch.int16, device=DEV)
        return s
    if kind == "timescales":
        cube, sigma, _ = _search_inputs(c, seed)
        scales = []
        for f, cfg in _scales(c):
            scales.append((f, native.Plan(cfg), sigma * math.sqrt(f)))
        return dict(kind=kind, cube=cube, scales=scales)
    if kind == "serve":
        eps = EPS if c["dtype"] != "f32" else 0.0
        plan = native.Plan(_config(c), dtype=c["dtype"], rescore_eps=eps)
        plan.stream_open(c["n_blk"])
        view = plan.stream_block()
        blocks = list(_serve_blocks(c, seed))
        for b in blocks[:-1]:
            view.copy_(b)
            plan.stream_push_device()
            plan.stream_poll(timeout_ms=20000)
        return dict(kind=kind, plan=plan, view=view, block=blocks[-1])
    if kind == "image":
        uv, chan, vis = _vis(c, seed)
        return dict(kind=kind, imager=native.Imager(uv, chan, n_grid=c["n_grid"]), vis=vis)
    if kind == "train":
        x, labels = _train_batch(c, seed)
        return dict(kind=kind, clf=_clf(c, c["c0"], c["batch"], seed, c["dropout"]), x=x, labels=labels)
    cfg = _config(dict(c, threshold=6.0))
    cube = synth.psf_noise(cfg, seed, device=DEV)
    return dict(kind=kind, plan=native.Plan(cfg), cube=cube, sigma=_sigma(c, cfg.n_pix), d=c["d"], hw=c["hw"],
                cands=native.candidates_to_device(_clf_cands(c, seed)),
                clf=_clf(c, c["n_sub"], c["n_cand"], seed, 0.5))


def _scales(c):
    return [(f, _config(c, n_t=c["n_t"] // f, factor=f, dm=dm, w_max=min(16, c["n_t"] // f)))
            for f, dm in ((5, 5.0 * np.linspace(0.0, c["dm_max"], c["n_dm"])), (75, np.array([0.0])))]


def _list(cand, n_pix):
    """The candidates in a table of one row per pixel (a pixel has one at most), zeros past the last."""
    table = np.zeros(n_pix, native.CANDIDATE_DTYPE)
    table[:len(cand)] = cand
    return {"n": len(cand), **{k: table[k] for k in FIELDS + ("snr",)}}


def run(s):
    kind = s["kind"]
    if kind == "search":
        plan = s["plan"]
        plan.search(s["cube"], s["sigma"], s["cube32"])
        if s["full"]:
            # the C entry point takes device buffers: the arrays stay on the GPU
            native._check(native.lib.nsfrb_full(plan.handle, s["snr"].data_ptr(), s["toa"].data_ptr()), "nsfrb_full")
            return {"snr": s["snr"], "toa": s["toa"]}
        return _list(plan.candidates(), plan.cfg.n_pix)
    if kind == "timescales":
        out = []
        for f, plan, sigma in s["scales"]:
            binned = multiscale.bin_time(s["cube"], f)
            plan.search(binned, sigma)
            out.append({"binned": binned, "found": _list(plan.candidates(), plan.cfg.n_pix)})
        return out
    if kind == "serve":
        s["view"].copy_(s["block"])
        s["plan"].stream_push_device()
        return _list(s["plan"].stream_poll(timeout_ms=20000)[0], s["plan"].cfg.n_pix)
    if kind == "image":
        return s["imager"].image(s["vis"])
    if kind == "train":
        loss = s["clf"].train_step(s["x"], s["labels"])
        return {"loss": loss, "grads": s["clf"].grads()}
    x = native.cutouts(s["plan"], s["cube"], s["cands"], s["d"], s["hw"], s["hw"], sigma=s["sigma"])
    return {"cutouts": x, "logits": s["clf"].infer(x)}


def _search_flops(n_pix, n_sub, n_t, rows, widths, last=0):
    """Per distinct DM row: the subbands whose shift changed (an add and a subtract per sample; the first row all
    subbands), one prefix add per sample, a difference and a maximum per trial."""
    n, prev = 0, None
    for s in rows:
        length = n_t - int(s.max())
        if length < 1:
            break
        n += length * (n_sub if prev is None else 2 * int((s != prev).sum())) + length
        for w in widths:
            n += 2 * max(0, min(length - w + 1, last or n_t))
        prev = s
    return float(n) * n_pix


def work(case):
    c, kind = case, case["kind"]
    es = 4 if c.get("dtype", "f32") == "f32" else 2
    if kind in ("search", "timescales", "serve"):
        n_pix = c["ny"] * c["nx"]
        samples = n_pix * c["n_sub"] * c["n_t"]
        rows = np.unique(_delays(np.linspace(0.0, c["dm_max"], c["n_dm"]), c["n_sub"]), axis=0)
    if kind == "search":
        widths = _widths(c["w_max"])
        bytes_ = samples * es + 4 * n_pix
        if c["out"] == "full":
            bytes_ += 6 * n_pix * c["n_dm"] * len(widths)
        return {"bytes": bytes_, "flops": _search_flops(n_pix, c["n_sub"], c["n_t"], rows, widths)}
    if kind == "timescales":
        flops = 2.0 * samples
        for (f, cfg), r in zip(_scales(c), (rows, np.zeros((1, c["n_sub"]), int))):
            flops += _search_flops(n_pix, c["n_sub"], cfg.n_t, r, cfg.widths)
        return {"bytes": samples * es + 4 * n_pix + sum(4 * n_pix * c["n_sub"] * (c["n_t"] // f) for f in (5, 75)),
                "flops": flops}
    if kind == "serve":
        # the block is read, the window is read once, the new samples are written
        blk = n_pix * c["n_sub"] * c["n_blk"]
        return {"bytes": samples * es + blk * (4 + es + (4 if es == 2 else 0)),
                "flops": _search_flops(n_pix, c["n_sub"], c["n_t"], rows, _widths(c["w_max"]), c["n_blk"])}
    if kind == "image":
        n_base = (c["n_ew"] + c["n_ns"]) * (c["n_ew"] + c["n_ns"] - 1) // 2
        n_vis = c["n_t"] * c["n_sub"] * c["n_chan"] * n_base
        n, img = c["n_grid"], c["n_t"] * c["n_sub"]
        return {"bytes": 16.0 * n_vis + 4.0 * img * n * n,
                "flops": 8.0 * n_vis + img * 10.0 * n * n * math.log2(n)}
    c0 = c["c0"] if kind == "train" else c["n_sub"]
    n = c["batch"] if kind == "train" else c["n_cand"]
    flops, cin, vox = 0.0, c0, c["d"] * c["hw"] ** 2
    for co in _chans(c):
        flops += 2.0 * vox * 27 * cin * co
        cin, vox = co, vox // 8
    x_bytes = 2.0 * n * c["d"] * c["hw"] ** 2 * c0
    if kind == "train":
        first = 2.0 * c["d"] * c["hw"] ** 2 * 27 * c0 * _chans(c)[0]
        return {"bytes": x_bytes + 4.0 * _clf_params(c, c0, 0).size, "flops": n * (3 * flops - first)}
    return {"bytes": 2 * x_bytes, "flops": n * flops}


# ------------------------------------------------------------------ the results in 64 bits

def _normalise64(x):
    """(x - median) / (1.4826 MAD) per row; rows of an even count take the mean of the two middle values."""
    n = x.shape[-1]

    def median(v):
        v = v.sort(dim=-1).values
        return 0.5 * (v[..., (n - 1) // 2] + v[..., n // 2])[..., None]

    x = x - median(x)
    return x / (1.4826 * median(x.abs()))


def _snr64(cube, sigma, n_sub, dm, t_samp, widths, mad=False, last=0, full=False):
    """Best S/N per pixel, or every (pixel, DM, width), of cube [n_pix, n_sub, n_t]."""
    n_pix, _, n_t = cube.shape
    rows, of_dm = np.unique(_delays(dm, n_sub, t_samp), axis=0, return_inverse=True)
    of_dm = torch.from_numpy(of_dm.reshape(-1)).to(DEV)
    best = torch.full((n_pix, len(dm), len(widths)) if full else (n_pix,), -math.inf, dtype=torch.float64, device=DEV)
    step = max(1, int(6e7 // (n_sub * n_t)))
    for p in range(0, n_pix, step):
        x = cube[p:p + step].double()
        m = x.shape[0]
        if mad:
            x = _normalise64(x)
            sg = torch.full((m,), math.sqrt(n_sub), dtype=torch.float64, device=DEV)
        else:
            sg = sigma[p:p + step].double()
        every = torch.full((m, len(rows), len(widths)), -math.inf, dtype=torch.float64, device=DEV)
        x = torch.nn.functional.pad(x, (0, int(rows.max())))
        prev = None
        for u, s in enumerate(rows):
            if prev is None:
                d = sum(x[:, k, s[k]:s[k] + n_t] for k in range(n_sub))
            else:
                for k in np.nonzero(s != prev)[0]:
                    d = d + (x[:, k, s[k]:s[k] + n_t] - x[:, k, prev[k]:prev[k] + n_t])
            prev = s
            length = n_t - int(s.max())
            if length < 1:
                continue
            sums = torch.zeros((m, length + 1), dtype=torch.float64, device=DEV)
            torch.cumsum(d[:, :length], 1, out=sums[:, 1:])
            for wi, w in enumerate(int(v) for v in widths):
                if w > length:
                    continue
                lo = max(0, length - w - last + 1) if last else 0
                every[:, u, wi] = (sums[:, w + lo:] - sums[:, lo:length + 1 - w]).amax(1) / (sg * math.sqrt(w))
        best[p:p + step] = every[:, of_dm] if full else every.amax((1, 2))
    return best


def _exact_list(best, threshold, rescored=None):
    if rescored is not None:
        best = torch.where((best - threshold).abs() <= EPS, rescored, best)
    found = best[best > threshold]
    snr = np.zeros(best.shape[0])
    snr[:found.numel()] = found.cpu().numpy()
    return {"n": None, **{k: None for k in FIELDS}, "snr": snr}


class _Stored(torch.autograd.Function):
    """BF16 storage of the value (forward) or of its gradient (backward): nearest even, kept in 64 bits."""

    @staticmethod
    def forward(ctx, v, back):
        ctx.back = back
        return v.clone() if back else v.to(torch.bfloat16).double()

    @staticmethod
    def backward(ctx, g):
        return (g.to(torch.bfloat16).double() if ctx.back else g), None


def _network64(c, p, x, keep=None, stats=None):
    """Logits of the classifier in 64 bits, with the network's own storage: its pooled activations and the gradients
    at the convolutions' outputs are BF16.  p: name -> tensor, x [B, d, h, w, c0]; batch statistics, or those given."""
    at = 0
    for l, co in enumerate(_chans(c)):
        b, d, h, w, ci = x.shape
        pad = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
        y = 0
        for tap in range(27):
            z, r = divmod(tap, 9)
            r, q = divmod(r, 3)
            y = y + pad[:, z:z + d, r:r + h, q:q + w].reshape(-1, ci) @ p["w%d" % l][:, tap].T
        y = _Stored.apply(y, True)
        if stats is None:
            mean, var = y.mean(0), y.var(0, unbiased=False)
        else:
            mean, var = stats[0][at:at + co], stats[1][at:at + co]
            at += co
        y = torch.relu((y - mean) / torch.sqrt(var + 1e-5) * p["g%d" % l] + p["b%d" % l])
        y = y.view(b, d // 2, 2, h // 2, 2, w // 2, 2, co).permute(0, 1, 3, 5, 7, 2, 4, 6).flatten(5)
        x = _Stored.apply(y.gather(5, y.detach().argmax(5, keepdim=True))[..., 0], False)
    hid = torch.relu(x.reshape(x.shape[0], -1) @ p["fw"].T + p["fb"])
    if keep is not None:
        hid = hid * keep
    return hid @ p["ow"] + p["ob"][0]


def _params64(c, c0, seed):
    flat = torch.from_numpy(_clf_params(c, c0, seed)).double().to(DEV).requires_grad_()
    p, o = {}, 0
    for name, shape in _clf_layout(c, c0):
        n = int(np.prod(shape))
        p[name] = flat[o:o + n].view(shape)
        o += n
    return flat, p


def _keep(n, f, rate, key):
    """The dropout mask of the first step: Philox4x32-10 words of counters (i, 0, 0, 0)."""
    lo = np.uint64(0xFFFFFFFF)
    x = [np.arange(n * f, dtype=np.uint64)] + [np.zeros(n * f, np.uint64) for _ in range(3)]
    k0, k1 = np.uint64(key & 0xFFFFFFFF), np.uint64(key >> 32)
    for _ in range(10):
        a, b = x[0] * np.uint64(0xD2511F53), x[2] * np.uint64(0xCD9E8D57)
        x = [(b >> np.uint64(32)) ^ x[1] ^ k0, b & lo, (a >> np.uint64(32)) ^ x[3] ^ k1, a & lo]
        k0, k1 = (k0 + np.uint64(0x9E3779B9)) & lo, (k1 + np.uint64(0xBB67AE85)) & lo
    u = (x[0] >> np.uint64(8)).astype(np.float64) * 2.0 ** -24
    return torch.from_numpy((u >= rate).astype(np.float64) / (1.0 - rate)).view(n, f).to(DEV)


def _cutouts64(c, cube, sigma, cands):
    """[n, d, h, w, n_sub]: bins of b samples around each candidate, over its pixel's noise per sample."""
    ny, nx, n_sub, n_t, d, hw = c["ny"], c["nx"], c["n_sub"], c["n_t"], c["d"], c["hw"]
    top = _delays(np.linspace(0.0, c["dm_max"], c["n_dm"]), n_sub).max(1)
    sums = torch.zeros((ny, nx, n_sub, n_t + 1), dtype=torch.float64, device=DEV)
    torch.cumsum(cube.double().view(ny, nx, n_sub, n_t), 3, out=sums[..., 1:])
    out = torch.zeros((len(cands), d, hw, hw, n_sub), dtype=torch.float64, device=DEV)
    for i, q in enumerate(cands):
        span = _widths(c["w_max"])[int(q["w_idx"])] + int(top[int(q["dm_idx"])])
        b = max(1, -(-span // (d // 2)))
        t = int(q["t_idx"]) + span // 2 - (d * b) // 2 + b * torch.arange(d + 1, device=DEV)
        t = t.clamp(0, n_t)
        r0, c0 = int(q["row"]) - hw // 2, int(q["col"]) - hw // 2
        a, e, f, g = max(r0, 0), min(r0 + hw, ny), max(c0, 0), min(c0 + hw, nx)
        box = sums[a:e, f:g][..., t]
        val = (box[..., 1:] - box[..., :-1]) / b / (sigma[int(q["row"]) * nx + int(q["col"])].double() / math.sqrt(n_sub))
        out[i, :, a - r0:e - r0, f - c0:g - c0] = val.permute(3, 0, 1, 2)
    return out


def _image64(c, uv, chan, vis, pixel_arcsec=10.3, robust=-2.0, b_min=20.0, b_max=485.0):
    n = c["n_grid"]
    half, mid = (n - 1) // 2, n // 2
    length = np.hypot(uv[:, 0], uv[:, 1])
    v = vis.to(torch.complex128).sum(-1)
    out = torch.empty((c["n_t"], c["n_sub"], n, n), dtype=torch.float64, device=DEV)
    for s in range(c["n_sub"]):
        grid = torch.zeros((c["n_t"], n * n), dtype=torch.complex128, device=DEV)
        for ch in range(c["n_chan"]):
            k = np.rint(uv * chan[s, ch] * 1.0e6 / C_LIGHT * n * (pixel_arcsec * math.pi / 648000.0)).astype(np.int64)
            ok = np.nonzero((length > b_min) & (length < b_max) & (np.abs(k) <= half).all(1))[0]
            here, there = (mid + k[ok, 1]) * n + mid + k[ok, 0], (mid - k[ok, 1]) * n + mid - k[ok, 0]
            count = np.bincount(np.concatenate([here, there]), minlength=n * n).astype(float)
            if not ok.size:
                continue
            f2 = (5.0 * 10.0 ** -robust) ** 2 / ((count ** 2).sum() / (2.0 * ok.size))
            wt = torch.from_numpy(1.0 / (1.0 + count[here] * f2)).to(DEV)
            val = v[:, s, ch][:, torch.from_numpy(ok).to(DEV)] * wt
            grid.index_add_(1, torch.from_numpy(here).to(DEV), val)
            grid.index_add_(1, torch.from_numpy(there).to(DEV), val.conj())
        z = torch.fft.ifftshift(grid.view(-1, n, n), dim=(1, 2))
        out[:, s] = torch.fft.ifftshift(torch.fft.ifft2(z), dim=(1, 2)).real
    return out


def exact(case, seed):
    c, kind = case, case["kind"]
    dm = np.linspace(0.0, c["dm_max"], c["n_dm"]) if "n_dm" in c else None
    if kind == "search":
        cube, sigma, cube32 = _search_inputs(c, seed)
        args = (sigma, c["n_sub"], dm, 134.2, _widths(c["w_max"]), c["noise"] == "mad")
        if c["out"] == "full":
            return {"snr": _snr64(cube, *args, full=True), "toa": None}
        best = _snr64(cube, *args)
        return _exact_list(best, c["threshold"], _snr64(cube32, *args) if c["rescore"] else None)
    if kind == "timescales":
        cube, sigma, _ = _search_inputs(c, seed)
        out = []
        for f, cfg in _scales(c):
            n = cfg.n_t * f
            x = torch.empty((cube.shape[0], c["n_sub"], cfg.n_t), dtype=torch.float64, device=DEV)
            for p in range(0, cube.shape[0], 4096):
                x[p:p + 4096] = cube[p:p + 4096, :, :n].double().view(-1, c["n_sub"], cfg.n_t, f).sum(-1)
            best = _snr64(x, sigma.double() * math.sqrt(f), c["n_sub"], cfg.dm, cfg.t_samp_ms, cfg.widths)
            out.append({"binned": x, "found": _exact_list(best, c["threshold"])})
        return out
    if kind == "serve":
        win = torch.cat([b.reshape(c["n_blk"], c["n_sub"], -1) for b in _serve_blocks(c, seed)])[-c["n_t"]:]
        sigma = torch.full((win.shape[2],), math.sqrt(c["n_sub"]), device=DEV)
        args = (sigma, c["n_sub"], dm, 134.2, _widths(c["w_max"]))
        cube = win.permute(2, 1, 0).contiguous()
        wide = _snr64(cube, *args, last=c["n_blk"]) if c["dtype"] != "f32" else None
        return _exact_list(_snr64(cube.to(_STORE[c["dtype"]]), *args, last=c["n_blk"]), c["threshold"], wide)
    if kind == "image":
        return _image64(c, *_vis(c, seed))
    if kind == "train":
        x, labels = _train_batch(c, seed)
        flat, p = _params64(c, c["c0"], seed)
        keep = _keep(c["batch"], c["f"], c["dropout"], 7)
        logits = _network64(c, p, x.double(), keep)
        loss = torch.nn.functional.binary_cross_entropy_with_logits(logits, labels.double())
        loss.backward()
        return {"loss": loss.detach().reshape(()), "grads": flat.grad}
    cfg = _config(dict(c, threshold=6.0))
    cube = synth.psf_noise(cfg, seed, device=DEV)
    x = _cutouts64(c, cube, _sigma(c, cfg.n_pix), _clf_cands(c, seed))
    _, p = _params64(c, c["n_sub"], seed)
    stats = [torch.from_numpy(v).double().to(DEV) for v in _bn_stats(c, seed)]
    with torch.no_grad():
        return {"cutouts": x, "logits": _network64(c, p, x, stats=stats)}
