"""The work a user has this library do, as cases that can be timed and compared.

Each case is one call, or one short series of calls, of the public entry
points of ``paper_1306_1467_gb300.vjb`` on seeded synthetic windows: whole
training jobs from the windows to the trained stumps, rounds on a training set
that is already prepared, batches, served requests, the strong classifier on
new windows, and the allocation-free search.  Sizes are those of the synthetic
workloads, the tests and the benchmark: windows from 10x10 to 32x32, training
sets from 600 windows to the limit of 32,766.
"""

from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_1306_1467_gb300 import vjb

DEV = "cuda"


# ---------------------------------------------------------------- the cases

def listed():
    return [
        # the smallest training run (10x10, 200 faces + 400 non-faces, 10
        # rounds): launches, copies and host work count, not bandwidth
        dict(name="job_10x10_600", kind="job", n=600, h=10, w=10, pos=1 / 3, rounds=10, source="host"),
        # the paper-shaped job: 24x24, 5000 faces + 10000 non-faces, all
        # 162,336 features, 200 rounds, windows already on the device
        dict(name="job_24x24_15000", kind="job", n=15000, h=24, w=24, pos=1 / 3, rounds=200, source="device"),
        # a retraining request's job: 24x24, a ragged sample count, 50 rounds,
        # windows on the host
        dict(name="job_24x24_10963", kind="job", n=10963, h=24, w=24, pos=0.35, rounds=50, source="host"),
        # the larger window of the served mix (32x32: 510,112 features), where
        # preparing the table weighs as much as the rounds
        dict(name="job_32x32_5003", kind="job", n=5003, h=32, w=32, pos=0.4, rounds=50, source="host"),
        # above 16,384 samples: 20x20 windows, the upper end of the batched
        # jobs' sample counts
        dict(name="job_20x20_19997", kind="job", n=19997, h=20, w=20, pos=0.25, rounds=50, source="device"),
        # training continued from given weights one round at a time, with the
        # per-feature errors of the last search: a short table, a call a round
        dict(name="rounds_24x24_2003", kind="rounds", n=2003, h=24, w=24, pos=0.4, rounds=8, single=True),
        # rounds at the largest training set the library takes
        dict(name="rounds_20x20_32766", kind="rounds", n=32766, h=20, w=20, pos=0.3, rounds=10, single=False),
        # a batch of uneven jobs (2,000 to 20,000 samples, 24x24) added,
        # trained together and removed
        dict(name="batch_24x24_8", kind="batch", jobs=8, n_lo=2000, n_hi=20000, h=24, w=24, rounds=40),
        # retraining requests of mixed window sizes, submitted together and
        # served until all are done
        dict(name="serve_mix_6", kind="serve", jobs=6, n_lo=2000, n_hi=8000, rounds=50),
        # the trained classifier on a handful of candidate windows, and on the
        # windows of a large scan
        dict(name="classify_24x24_200", kind="classify", n=200, h=24, w=24, stumps=200),
        dict(name="classify_24x24_150001", kind="classify", n=150001, h=24, w=24, stumps=200),
        # the allocation-free search over a caller's own table (16x16, 15,000
        # samples: a table above the L2 cache)
        dict(name="noalloc_16x16_15000", kind="noalloc", n=15000, h=16, w=16, pos=1 / 3),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["job", "job", "job", "rounds", "rounds", "batch", "serve", "classify", "classify", "noalloc"])
    if kind == "batch":
        return dict(kind=kind, jobs=rng.randint(2, 8), n_lo=2000, n_hi=_log_int(rng, 4000, 20000), h=24, w=24,
                    rounds=_log_int(rng, 8, 40))
    if kind == "serve":
        return dict(kind=kind, jobs=rng.randint(2, 6), n_lo=2000, n_hi=_log_int(rng, 3000, 8000),
                    rounds=_log_int(rng, 10, 50))
    if kind == "classify":
        h = rng.randint(10, 32)
        return dict(kind=kind, n=_log_int(rng, 1, 150000), h=h, w=rng.choice([h, h, rng.randint(10, 32)]),
                    stumps=_log_int(rng, 1, 200))
    most = 5e8 if kind == "noalloc" else 2.6e9  # features x samples
    while True:
        h = rng.randint(10, 32)
        w = rng.choice([h, h, rng.randint(10, 32)])
        n = _log_int(rng, 600, 32766)
        if feature_count(h, w) * n <= most:
            break
    c = dict(kind=kind, n=n, h=h, w=w, pos=rng.uniform(0.2, 0.5))
    if kind == "job":
        # at most the work of the paper-shaped job
        top = int(min(200, 5e11 / (feature_count(h, w) * n) - 28))
        c.update(rounds=_log_int(rng, min(10, top), top), source=rng.choice(["host", "device"]))
    elif kind == "rounds":
        c.update(rounds=_log_int(rng, 1, 20), single=rng.random() < 0.5)
    return c


def work(case):
    """What one pass cannot do without.  Training holds the samples' order per
    feature (2 bytes per feature and sample): preparing a set writes it once,
    each round reads it once and adds one weight per entry."""
    k = case["kind"]
    if k == "classify":
        n, T = case["n"], case["stumps"]
        return {"bytes": n * case["h"] * case["w"] + 9.0 * n + 40.0 * T, "flops": 10.0 * n * T}
    if k == "noalloc":
        e = float(feature_count(case["h"], case["w"])) * case["n"]
        return {"bytes": 2 * e + 4.0 * case["n"] + 4.0 * feature_count(case["h"], case["w"]), "flops": e}
    by = fl = 0.0
    for s in _job_shapes(case, 0):
        e = float(feature_count(s["h"], s["w"])) * s["n"]
        fresh = k != "rounds"
        by += 2 * e * (s["rounds"] + fresh) + 4.0 * s["n"] + (s["n"] * (s["h"] * s["w"] + 1.0) if fresh else 4.0 * s["n"])
        fl += e * s["rounds"]
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------- inputs

def _blur(h, sigma):
    """[k, h, h] matrices of a reflecting Gaussian blur, one for each of k sigmas."""
    r = 9
    d = torch.arange(-r, r + 1, device=DEV)
    g = torch.exp(-0.5 * (d[None, :] / sigma[:, None]) ** 2)
    g = g / g.sum(1, keepdim=True)
    i = torch.arange(h, device=DEV)[None, :] + d[:, None]
    i = torch.remainder(i, 2 * h)
    i = torch.where(i >= h, 2 * h - 1 - i, i)
    hot = torch.nn.functional.one_hot(i, h).to(g.dtype)  # [2r + 1, h, h]
    return (g @ hot.reshape(2 * r + 1, h * h)).reshape(-1, h, h)


def windows(n, h, w, pos, seed):
    """uint8 windows [n, h, w] and labels [n] on the GPU, shaped like the
    synthetic training sets: faces a dark band over a bright band under strong
    smoothed noise, non-faces smoothed uniform noise."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    n_pos = max(1, min(n - 1, int(round(pos * n))))
    n_neg = n - n_pos
    one = torch.ones(1, device=DEV)
    t = torch.full((h, w), 128.0, device=DEV)
    t[h // 4: h // 2] = 64.0
    t[h // 2: (3 * h) // 4] = 192.0
    c = torch.rand(n_pos, 1, 1, generator=g, device=DEV) * 0.6 + 0.7
    o = torch.rand(n_pos, 1, 1, generator=g, device=DEV) * 40.0 - 20.0
    z = torch.randn(n_pos, h, w, generator=g, device=DEV) * 800.0
    z = _blur(h, one)[0] @ z @ _blur(w, one)[0].T
    faces = 128.0 + c * (t - 128.0) + o + z
    sig = torch.rand(n_neg, generator=g, device=DEV) * 2.5 + 0.5
    u = torch.rand(n_neg, h, w, generator=g, device=DEV) * 255.0
    rest = torch.bmm(torch.bmm(_blur(h, sig), u), _blur(w, sig).transpose(1, 2))
    px = torch.cat([faces, rest]).round().clamp(0, 255).to(torch.uint8)
    y = torch.cat([torch.ones(n_pos, dtype=torch.uint8, device=DEV), torch.zeros(n_neg, dtype=torch.uint8, device=DEV)])
    p = torch.randperm(n, generator=g, device=DEV)
    return px[p].contiguous(), y[p].contiguous()


def _weights(n, seed):
    """Weights of a run that goes on: spread over a factor of about 400."""
    rng = np.random.Generator(np.random.PCG64(int(seed)))
    return np.exp(rng.uniform(-3.0, 3.0, size=n)).astype(np.float32)


def _job_shapes(case, seed):
    """The training jobs of a case: dicts of n, h, w, pos, rounds and a seed of their own.
    The sizes follow from the case alone, the windows from the seed."""
    if case["kind"] in ("job", "rounds"):
        return [dict(n=case["n"], h=case["h"], w=case["w"], pos=case["pos"], rounds=case["rounds"], seed=seed)]
    out = []
    rng = np.random.Generator(np.random.PCG64(case["jobs"] * 100003 + case["n_hi"]))
    for k in range(case["jobs"]):
        n = int(rng.integers(case["n_lo"], case["n_hi"] + 1))
        if case["kind"] == "serve":  # most requests 24x24, some 20x20 and 32x32
            side = (24, 20, 24, 32, 24, 24)[k % 6]
            if side == 32:
                n = min(n, 4000)
            h = w = side
        else:
            h, w = case["h"], case["w"]
        out.append(dict(n=n, h=h, w=w, pos=float(rng.uniform(0.2, 0.5)), rounds=case["rounds"], seed=seed * 64 + k))
    return out


def _host(px, y):
    return px.cpu().numpy(), y.cpu().numpy()


def prepare(case, seed):
    k = case["kind"]
    s = dict(case)
    if k == "job":
        px, y = windows(case["n"], case["h"], case["w"], case["pos"], seed)
        s["px"], s["y"] = (px, y) if case["source"] == "device" else _host(px, y)
        s["trainer"] = vjb.Trainer()
    elif k == "rounds":
        px, y = windows(case["n"], case["h"], case["w"], case["pos"], seed)
        s["trainer"] = vjb.Trainer()
        s["trainer"].prepare(px, y)
        s["w0"] = _weights(case["n"], seed)
    elif k in ("batch", "serve"):
        shapes = _job_shapes(case, seed)
        s["data"] = [(*_host(*windows(j["n"], j["h"], j["w"], j["pos"], j["seed"])), j["rounds"]) for j in shapes]
        budget = sum(vjb.Batch.table_bytes(j["n"], j["h"], j["w"]) for j in shapes)
        s["engine"] = vjb.Batch(budget) if k == "batch" else vjb.Server(budget, max_jobs=16)
    elif k == "classify":
        px, y = windows(1000, case["h"], case["w"], 0.4, seed)
        s["trainer"] = vjb.Trainer()
        s["trainer"].prepare(px, y)
        _, s["strong"] = s["trainer"].train_strong(case["stumps"])
        s["px"] = _host(*windows(max(case["n"], 2), case["h"], case["w"], 0.1, seed + 1))[0][: case["n"]]
    elif k == "noalloc":
        px, y = windows(case["n"], case["h"], case["w"], case["pos"], seed)
        n, npad = case["n"], -(-case["n"] // 64) * 64
        F = feature_count(case["h"], case["w"])
        rows = torch.full((F, npad), n, dtype=torch.int16, device=DEV)
        for f0, order, valid in _orders(px):
            rows[f0: f0 + order.shape[0], :n] = order | torch.where(valid, -32768, 0).to(torch.int16)
        wt = torch.from_numpy(_weights(n, seed)).to(DEV)
        wt = wt / wt.sum()
        v = torch.zeros(n + 1, device=DEV)
        v[:n] = torch.where(y > 0, wt, -wt)
        s.update(rows=rows, v=v, npad=npad, F=F, t_pos=float(v[:n].clamp(min=0).double().sum()),
                 t_neg=float((-v[:n]).clamp(min=0).double().sum()), err=torch.empty(F, device=DEV),
                 best=torch.empty(1, device=DEV), at=torch.empty(1, dtype=torch.int32, device=DEV))
    return s


# ---------------------------------------------------------------- one pass

def _stumps(stumps):
    return {k: np.array([s[k] for s in stumps], np.int32 if k in ("feature", "threshold", "polarity", "split") else np.float64)
            for k in ("feature", "threshold", "polarity", "split", "error", "beta", "alpha")}


def run(s):
    k = s["kind"]
    if k == "job":
        tr = s["trainer"]
        feats = tr.prepare(s["px"], s["y"])
        status, stumps = tr.train_strong(s["rounds"])
        return {"features": feats, "status": status, "stumps": _stumps(stumps), "weights": tr.get_weights()}
    if k == "rounds":
        tr = s["trainer"]
        tr.set_weights(s["w0"])
        if s["single"]:
            got = [tr.train_round() for _ in range(s["rounds"])]
            status, stumps = got[-1][0], [g[1] for g in got]
        else:
            status, stumps = tr.train_strong(s["rounds"])
        return {"status": status, "stumps": _stumps(stumps), "weights": tr.get_weights(), "errors": tr.screen_errors()}
    if k == "batch":
        b = s["engine"]
        ids = [b.add_job(px, y, rounds) for px, y, rounds in s["data"]]
        b.train()
        out = [{"status": b.job_state(i)[1], "stumps": _stumps(b.stumps(i)), "weights": b.get_weights(i)} for i in ids]
        for i in ids:
            b.remove_job(i)
        return _flat(out)
    if k == "serve":
        srv = s["engine"]
        ids = [srv.submit(px, y, rounds) for px, y, rounds in s["data"]]
        while any(srv.request(i)["state"] not in (vjb.REQ_DONE, vjb.REQ_FAILED) for i in ids):
            srv.step(8)
        out = []
        for i in ids:
            status, stumps, w = srv.result(i)
            srv.release(i)
            out.append({"status": status, "stumps": _stumps(stumps), "weights": w})
        return _flat(out)
    if k == "classify":
        labels, scores = s["trainer"].classify(s["px"], s["strong"])
        return {"labels": labels, "scores": scores}
    lib = vjb.load_library()
    rc = lib.vjb_screen_noalloc(*(ctypes.c_void_p(s[x].data_ptr()) for x in ("rows", "v")), s["n"], s["npad"], s["F"],
                                s["t_pos"], s["t_neg"], 0, *(ctypes.c_void_p(s[x].data_ptr()) for x in ("err", "best", "at")),
                                ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    if rc != vjb.OK:
        raise vjb.VJBError(rc, lib.vjb_last_error().decode())
    return {"errors": s["err"], "best": s["best"], "at": s["at"]}


def _flat(jobs):
    """The jobs' results end to end, job after job (None where a job's value has none)."""
    def cat(parts):
        return None if any(p is None for p in parts) else np.concatenate([np.asarray(p) for p in parts])
    return {"status": cat([None if j["status"] is None else [j["status"]] for j in jobs]),
            "stumps": {k: cat([j["stumps"][k] for j in jobs]) for k in jobs[0]["stumps"]},
            "weights": cat([j["weights"] for j in jobs])}


# ---------------------------------------------------------------- the same in 64 bits

# per type: its base size, and its rectangles as (sign, x, y, w, h) in units of the base
_BASE = ((3, 1), (1, 3), (2, 1), (1, 2), (2, 2))
_RECTS = (((1, 1, 0), (-1, 0, 0), (-1, 2, 0)), ((1, 0, 1), (-1, 0, 0), (-1, 0, 2)), ((1, 1, 0), (-1, 0, 0)),
          ((1, 0, 1), (-1, 0, 0)), ((1, 1, 0), (1, 0, 1), (-1, 0, 0), (-1, 1, 1)))


def feature_count(h, w):
    return sum(sum(w - fw + 1 for fw in range(bw, w + 1, bw)) * sum(h - fh + 1 for fh in range(bh, h + 1, bh))
               for bw, bh in _BASE)


def _features(h, w):
    """[F, 5] (type, x, y, w, h): types in the order above, then width, height, y, x ascending."""
    out = []
    for t, (bw, bh) in enumerate(_BASE):
        for fw in range(bw, w + 1, bw):
            for fh in range(bh, h + 1, bh):
                y, x = np.mgrid[0: h - fh + 1, 0: w - fw + 1]
                out.append(np.stack([np.full(x.size, t), x.ravel(), y.ravel(), np.full(x.size, fw), np.full(x.size, fh)], 1))
    return np.concatenate(out)


def _integral(px):
    """int32 [(h + 1) * (w + 1), n] sums of the pixels above and left of each point."""
    n, h, w = px.shape
    ii = torch.zeros(n, h + 1, w + 1, dtype=torch.int32, device=px.device)
    ii[:, 1:, 1:] = px.to(torch.int32).cumsum(1).cumsum(2).to(torch.int32)
    return ii.reshape(n, -1).T.contiguous()


def _values(ii, w, feats):
    """int32 [len(feats), n] values of features that share one type."""
    t = int(feats[0, 0])
    x, y, fw, fh = (torch.from_numpy(np.ascontiguousarray(feats[:, k])).to(ii.device) for k in range(1, 5))
    a, b = fw // _BASE[t][0], fh // _BASE[t][1]
    v = None
    for sign, rx, ry in _RECTS[t]:
        for s, px, py in ((1, rx + 1, ry + 1), (1, rx, ry), (-1, rx + 1, ry), (-1, rx, ry + 1)):
            term = ii[(y + py * b) * (w + 1) + x + px * a]
            v = term * (sign * s) if v is None else v.add_(term, alpha=sign * s)
    return v


def _orders(px):
    """Blocks (first feature, samples in value order int16, split allowed after each) over all features."""
    n, h, w = px.shape
    ii, feats = _integral(px), _features(h, w)
    step = max(1, int(6e7 // n))
    ends = np.flatnonzero(np.diff(feats[:, 0])) + 1
    for lo, hi in zip([0, *ends], [*ends, len(feats)]):
        for f0 in range(lo, hi, step):
            vals, order = torch.sort(_values(ii, w, feats[f0: min(hi, f0 + step)]), dim=1, stable=True)
            valid = torch.ones_like(vals, dtype=torch.bool)
            valid[:, :-1] = vals[:, :-1] < vals[:, 1:]
            yield f0, order.to(torch.int16), valid


def _scan(v, order, valid):
    """Weight prefixes at the allowed splits: (largest, its split, smallest, its split), split 0 included."""
    D = torch.cumsum(v[order.long()], 1)
    mx, ax = torch.where(valid, D, -math.inf).max(1)
    mn, an = torch.where(valid, D, math.inf).min(1)
    return mx.clamp(min=0.0), torch.where(mx > 0, ax + 1, 0), mn.clamp(max=0.0), torch.where(mn < 0, an + 1, 0)


def _boost(px, y, w, rounds):
    """Discrete AdaBoost in 64 bits: the layout of run() for one job, with its last search's errors."""
    blocks = list(_orders(px))
    face = y > 0
    w = w / w.sum()
    out = {k: [] for k in ("error", "beta", "alpha")}
    for _ in range(rounds):
        v = torch.where(face, w, -w)
        tp, tn = w[face].sum(), w[~face].sum()
        best, errs = None, []
        for _, order, valid in blocks:
            mx, ax, mn, an = _scan(v, order, valid)
            plus, minus = tp - mx, tn + mn
            e = torch.minimum(plus, minus)
            errs.append(e)
            f = int(e.argmin())
            if best is None or float(e[f]) < best[0]:
                up = bool(plus[f] <= minus[f])
                s = int(ax[f] if up else an[f])
                below = torch.zeros_like(face)
                below[order[f, :s].long()] = True
                best = (float(e[f]), below if up else ~below)
        miss = best[1] != face
        eps = float(w[miss].sum() / w.sum())
        if not 0.0 < eps < 0.5:
            return None
        out["error"].append(eps)
        out["beta"].append(eps / (1 - eps))
        out["alpha"].append(math.log((1 - eps) / eps))
        w = torch.where(miss, w, w * out["beta"][-1])
        w = w / w.sum()
    st = {k: None for k in ("feature", "threshold", "polarity", "split")}
    st.update({k: np.array(a) for k, a in out.items()})
    return {"status": None, "stumps": st, "weights": w.cpu().numpy(), "errors": torch.cat(errs).cpu().numpy()}


def exact(case, seed):
    k = case["kind"]
    if k == "classify":
        s = prepare(case, seed)
        feats = _features(case["h"], case["w"])
        ii = _integral(torch.from_numpy(s["px"]).to(DEV))
        score = torch.zeros(case["n"], dtype=torch.float64, device=DEV)
        for c in s["strong"]:
            v = _values(ii, case["w"], feats[c["feature"]: c["feature"] + 1])[0]
            score += c["alpha"] * (c["polarity"] * v < c["polarity"] * c["threshold"]).double()
        return {"labels": None, "scores": score.cpu().numpy()}
    if k == "noalloc":
        s = prepare(case, seed)
        n, v, parts = case["n"], s["v"].double(), []
        for f0 in range(0, s["F"], max(1, int(6e7 // n))):
            r = s["rows"][f0: f0 + max(1, int(6e7 // n)), :n]
            mx, _, mn, _ = _scan(v, r & 32767, r < 0)
            parts.append(torch.minimum(s["t_pos"] - mx, s["t_neg"] + mn))
        e = torch.cat(parts)
        return {"errors": e, "best": e.min().reshape(1), "at": None}
    shapes = _job_shapes(case, seed)
    # sorting costs about ten rounds' scans; over this it takes longer than 20 s
    if sum(feature_count(j["h"], j["w"]) * j["n"] * (j["rounds"] + 10.0) for j in shapes) > 6e10:
        return None
    out = []
    for j in shapes:
        px, y = windows(j["n"], j["h"], j["w"], j["pos"], j["seed"])
        if k == "rounds":
            w = torch.from_numpy(_weights(j["n"], j["seed"])).to(DEV).double()
        else:
            w = torch.where(y > 0, 0.5 / (y > 0).sum(), 0.5 / (y == 0).sum()).double()
        got = _boost(px, y, w, j["rounds"])
        if got is None:
            return None
        out.append(got)
    if k == "rounds":
        return out[0]
    if k == "job":
        return {"features": None, **{x: out[0][x] for x in ("status", "stumps", "weights")}}
    return _flat(out)
