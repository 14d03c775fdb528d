"""The work whose time is watched: what a user of this library has it do.

Every case goes through the package's public entry points on inputs shaped
like the workloads of ``synth`` and ``bench.py`` (uniform, seasonal and nightly
cadences over ten years, sinusoid plus noise), from one short light curve
to batches of tens of thousands.

A case is a dict of plain values.  ``kind`` names the entry point:

* ``single``  -- ``periodogram``: one light curve, full power array and peaks;
* ``batch``   -- ``batch``: a ragged CSR batch, peaks and optionally all powers;
* ``plan``    -- ``Plan.execute``: the same batch as a prepared, graph-replayed job;
* ``host``    -- ``Plan.execute_host``: from page-locked host buffers, peaks back;
* ``gls``     -- ``batch_gls``: errors and a floating mean;
* ``learned`` -- ``LearnedPath``: proposal network, refine, full-grid fallback;
* ``train``   -- ``Proposer.train_step``: loss, gradients and the AdamW update.
"""
import math
import os

import numpy as np
import torch

import paper_2105_04006_gb300 as lsp
from paper_2105_04006_gb300 import learned

DEV = "cuda"
SPAN = 3652.5  # ten years, in days


def listed():
    return [
        # one short light curve on a coarse grid, as in an interactive look: latency and launches
        {"name": "single_quick", "kind": "single", "n_t": 120, "n_f": 5000, "f_min": 0.1, "f_max": 5.0,
         "precision": "fp32", "cadence": "uniform", "top_k": 1, "norm": "standard"},
        # the single-object workload (synth.single_small), both precisions
        {"name": "single_small", "kind": "single", "n_t": 1000, "n_f": 100_000, "f_min": 0.1, "f_max": 10.0,
         "precision": "fp32", "cadence": "uniform", "top_k": 1, "norm": "standard"},
        {"name": "single_small_fp64", "kind": "single", "n_t": 1000, "n_f": 100_000, "f_min": 0.1, "f_max": 10.0,
         "precision": "fp64", "cadence": "uniform", "top_k": 1, "norm": "standard"},
        # one well-observed object on a long grid (synth.single_large), and its FP64 form at half the size
        {"name": "single_large", "kind": "single", "n_t": 100_000, "n_f": 1_000_000, "f_min": 0.05, "f_max": 25.0,
         "precision": "fp32", "cadence": "uniform", "top_k": 1, "norm": "standard"},
        {"name": "single_large_fp64", "kind": "single", "n_t": 50_000, "n_f": 500_000, "f_min": 0.05, "f_max": 12.5,
         "precision": "fp64", "cadence": "uniform", "top_k": 1, "norm": "standard"},
        # the sparse survey batch (synth.ragged_survey) end to end from host memory: one period per object
        {"name": "survey_host", "kind": "host", "n_obj": 10_000, "nt_lo": 50, "nt_hi": 500, "log_nt": False,
         "n_f": 100_000, "f_min": 0.24, "f_max": 12.0, "precision": "fp32", "cadence": "seasonal", "top_k": 1,
         "norm": "standard"},
        # the lognormal batch (synth.ragged_lognormal's shape), three peaks per object, as a prepared plan
        {"name": "lognormal_top3", "kind": "plan", "n_obj": 20_000, "nt_lo": 10, "nt_hi": 2000, "log_nt": True,
         "n_f": 50_000, "f_min": 0.24, "f_max": 12.0, "precision": "fp32", "cadence": "seasonal", "top_k": 3,
         "norm": "standard"},
        # a night's alerts with every periodogram returned, in units of y^2, on an odd grid
        {"name": "alerts_power", "kind": "batch", "n_obj": 1000, "nt_lo": 50, "nt_hi": 500, "log_nt": False,
         "n_f": 100_003, "f_min": 0.24, "f_max": 12.0, "precision": "fp32", "cadence": "seasonal", "top_k": 1,
         "norm": "psd", "power": True},
        # a small batch in FP64: candidates re-examined at full precision
        {"name": "candidates_fp64", "kind": "batch", "n_obj": 200, "nt_lo": 50, "nt_hi": 500, "log_nt": False,
         "n_f": 100_000, "f_min": 0.24, "f_max": 12.0, "precision": "fp64", "cadence": "seasonal", "top_k": 1,
         "norm": "standard", "power": False},
        # the generalized periodogram (photometric errors, floating mean) of a survey batch
        {"name": "gls_survey", "kind": "gls", "n_obj": 2000, "nt_lo": 50, "nt_hi": 500, "log_nt": False,
         "n_f": 100_000, "f_min": 0.24, "f_max": 12.0, "precision": "fp32", "cadence": "seasonal", "top_k": 1,
         "norm": "standard", "power": False},
        # the learned path with the committed network on a survey batch
        {"name": "learned_survey", "kind": "learned", "n_obj": 20_000, "nt_lo": 50, "nt_hi": 500, "log_nt": False,
         "n_f": 100_000, "f_min": 0.24, "f_max": 12.0, "precision": "fp32", "cadence": "seasonal"},
        # one optimizer step of the proposal network at its training batch size
        {"name": "train_step", "kind": "train", "batch": 4096, "n_f": 100_000},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges; never more work than the largest listed one."""
    kind = rng.choice(["single", "single", "single", "plan", "host", "batch", "batch", "gls", "learned", "train"])
    if kind == "train":
        return {"kind": "train", "batch": _log_int(rng, 128, 16384), "n_f": rng.choice([50_000, 100_000])}
    if kind == "learned":
        return {"kind": "learned", "n_obj": _log_int(rng, 500, 20_000), "nt_lo": 50, "nt_hi": 500, "log_nt": False,
                "n_f": 100_000, "f_min": 0.24, "f_max": 12.0, "precision": "fp32", "cadence": "seasonal"}
    fp64 = rng.random() < 0.3
    c = {"kind": kind, "f_min": round(rng.uniform(0.05, 0.3), 3), "f_max": round(rng.uniform(4.0, 12.5), 2),
         "precision": "fp64" if fp64 else "fp32", "cadence": rng.choice(["uniform", "seasonal", "seasonal", "nightly"]),
         "top_k": rng.choice([1, 1, 3]), "norm": rng.choice(["standard", "standard", "psd"])}
    if kind == "single":
        c["n_t"] = _log_int(rng, 60, 50_000)
        most = 2.5e10 / c["n_t"] if fp64 else 1e11 / c["n_t"]
        c["n_f"] = _log_int(rng, 3000, min(500_000, most))
        if c["cadence"] == "nightly" and c["n_t"] > 3000:
            c["cadence"] = "uniform"  # at most one observation a night over ten years
        return c
    c["nt_lo"], c["nt_hi"], c["log_nt"] = rng.choice([(50, 500, False), (10, 2000, True)])
    c["n_f"] = _log_int(rng, 20_000, 120_000)
    pairs = (275 if not c["log_nt"] else 376) * c["n_f"]
    budget = 5e9 if fp64 else 1e11
    c["n_obj"] = max(4, min(_log_int(rng, 20, 8000), int(budget / pairs)))
    if kind in ("batch", "gls"):
        c["power"] = rng.random() < 0.5
        if c["power"]:
            c["n_obj"] = min(c["n_obj"], int(1e8 / c["n_f"]))
    return c


# ------------------------------------------------------------------- inputs
def _counts(case, g):
    """Observations per object (host list, so that sizes are known without a copy back)."""
    if case["kind"] == "single":
        return np.array([case["n_t"]], dtype=np.int64)
    r = np.random.default_rng(g.initial_seed())
    lo, hi, n = case["nt_lo"], case["nt_hi"], case["n_obj"]
    if case["log_nt"]:
        return np.rint(np.exp(r.uniform(math.log(lo), math.log(hi), n))).astype(np.int64)
    return r.integers(lo, hi + 1, n)


def _light_curves(case, seed):
    """t, y, dy (float64), offsets of a CSR batch on the GPU, sorted in time within each object."""
    g = torch.Generator(device=DEV).manual_seed(seed * 7919 + 13)
    n_t = _counts(case, g)
    off = np.concatenate([[0], np.cumsum(n_t)]).astype(np.int64)
    total, n_obj = int(off[-1]), len(n_t)
    u = lambda n: torch.rand(n, generator=g, device=DEV, dtype=torch.float64)  # noqa: E731
    obj = torch.repeat_interleave(torch.arange(n_obj, device=DEV), torch.from_numpy(n_t).to(DEV), output_size=total)
    if case["cadence"] == "seasonal":  # six months of every year
        t = torch.floor(u(total) * 10) * 365.25 + u(total) * 182.625
    elif case["cadence"] == "nightly":  # within one hour of a night
        t = torch.floor(u(total) * 3650) + 0.3 + u(total) / 24
    else:
        t = u(total) * SPAN
    key, _ = torch.sort(obj.double() * 4096.0 + t)
    t = 60000.0 + (key - obj.double() * 4096.0)
    sigma = 0.02 + 0.28 * u(n_obj)
    f0 = 24.0 / torch.exp(math.log(2.0) + u(n_obj) * math.log(50.0))  # periods of 2 to 100 hours
    f0 = torch.minimum(f0, torch.full_like(f0, 0.9 * case["f_max"]))
    ph = 2 * math.pi * u(n_obj)
    noise = torch.randn(total, generator=g, device=DEV, dtype=torch.float64)
    dy = sigma[obj] * (0.5 + u(total))
    y = 15.0 + 0.5 * torch.sin(2 * math.pi * torch.frac(f0[obj] * t) + ph[obj]) + noise * dy
    dt = torch.float64 if case["precision"] == "fp64" else torch.float32
    return t, y.to(dt), dy.to(dt), torch.from_numpy(off).to(DEV)


def _grid(case):
    return lsp.Grid(case["f_min"], case["f_max"], case["n_f"])


def _net():
    path = os.path.join(os.path.dirname(learned.__file__), "weights", "proposer_survey.npz")
    return learned.Proposer.load_npz(path, DEV)[0]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        g = torch.Generator(device=DEV).manual_seed(seed * 7919 + 29)
        net = learned.Proposer(case["n_f"], DEV, seed=1 + seed % 1000)
        x = 0.3 * torch.randn((case["batch"], learned.FEAT_DIM), generator=g, device=DEV)
        lab = torch.randint(0, net.dims.n_classes, (case["batch"],), generator=g, device=DEV, dtype=torch.int32)
        return {"case": case, "net": net, "x": x.to(torch.bfloat16), "labels": lab}
    t, y, dy, off = _light_curves(case, seed)
    s = {"case": case, "grid": _grid(case), "t": t, "y": y, "dy": dy, "off": off}
    s["opts"] = {k: case[k] for k in ("precision", "norm", "top_k") if k in case}
    n_obj = off.numel() - 1
    if kind in ("plan", "host"):
        s["plan"] = lsp.Plan(n_obj, t.numel(), s["grid"], **s["opts"])
        if kind == "plan":
            s["peaks"] = s["plan"].peaks_buffer(t.device)
        else:
            s["host"] = [a.cpu().pin_memory() for a in (t, y, off)]
            s["peaks"] = torch.empty(n_obj * case["top_k"] * 40, dtype=torch.uint8).pin_memory()
    elif kind == "learned":
        s["path"] = learned.LearnedPath(_net())
        s["classes"] = torch.empty((n_obj, s["path"].proposer.k_windows), dtype=torch.int32, device=DEV)
    return s


# --------------------------------------------------------------------- pass
def _decode(peaks, top_k, precision):
    """The fields of 40-byte peak records; an FP32 call's powers are FP32 values stored wide."""
    w, f = peaks.view(torch.int64).view(-1, top_k, 5), peaks.view(torch.float64).view(-1, top_k, 5)
    power = f[..., 1] if precision == "fp64" else f[..., 1].float()
    return {"idx": w[..., 0], "peak_power": power, "freq_period": f[..., 2:4], "flags": w[..., 4]}


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "train":
        net = s["net"]
        loss = net.train_step(s["x"], s["labels"])
        return {"loss": loss, "grad": net.grad, "params": net.params, "m": net.m, "v": net.v}
    if kind == "learned":
        peaks, info = s["path"](s["t"], s["y"], s["off"], s["grid"], classes_out=s["classes"])
        return dict(_decode(peaks, 1, "fp32"), info=info, classes=s["classes"])
    power = None
    if kind == "single":
        power, peaks = lsp.periodogram(s["t"], s["y"], s["grid"], **s["opts"])
    elif kind == "batch":
        power, peaks = lsp.batch(s["t"], s["y"], s["off"], s["grid"], return_power=case["power"], **s["opts"])
    elif kind == "gls":
        power, peaks = lsp.batch_gls(s["t"], s["y"], s["dy"], s["off"], s["grid"], return_power=case["power"],
                                     **s["opts"])
    elif kind == "plan":
        peaks = s["plan"].execute(s["t"], s["y"], s["off"], peaks=s["peaks"])
    else:
        peaks = s["plan"].execute_host(*s["host"], peaks=s["peaks"])
    out = _decode(peaks, case["top_k"], case["precision"])
    if power is not None:
        out["power"] = power
    return out


# ------------------------------------------------------------ what it takes
def _mean_total(case):
    if case["kind"] == "single":
        return case["n_t"]
    lo, hi = case["nt_lo"], case["nt_hi"]
    return case["n_obj"] * ((hi - lo) / math.log(hi / lo) if case["log_nt"] else 0.5 * (lo + hi))


def work(case):
    """Each input read once, each output written once; operations of the least known way there: two (with
    errors: three) fast transforms of every grid, 30 operations a bin for its power, 50 an observation."""
    if case["kind"] == "train":
        c = learned.n_classes(case["n_f"])
        macs = case["batch"] * (512 * 256 + 2 * 256 * 256 + 256 * c)
        n_par = 512 * 256 + 256 + 2 * (256 * 256 + 256) + 256 * c + c
        # read x, labels, p, m, v; write grad, p, m, v, the 16-bit copy; forward, weight and input gradients
        return {"bytes": case["batch"] * (1024 + 4) + n_par * (3 * 4 + 4 * 4 + 2),
                "flops": 2 * (3 * macs - case["batch"] * 512 * 256)}
    total = _mean_total(case)
    n_obj = case.get("n_obj", 1)
    el = 8 if case["precision"] == "fp64" else 4
    n_in = total * (8 + el * (2 if case["kind"] == "gls" else 1)) + 8 * (n_obj + 1)
    if case["kind"] == "learned":
        # the pairs of the features, the network, one refined window and one in twenty objects on the full grid
        net = 512 * 256 + 2 * 256 * 256 + 256 * learned.n_classes(case["n_f"])
        per = 2 * net + 2048 * 250 + 0.05 * case["n_f"] * 200
        return {"bytes": n_in + n_obj * (40 + 4 + 32), "flops": n_obj * per + 50 * total}
    transforms = 3 if case["kind"] == "gls" else 2
    flops = n_obj * case["n_f"] * (5 * transforms * math.log2(2 * case["n_f"]) + 30) + 50 * total
    power = case["kind"] == "single" or case.get("power", False)
    return {"bytes": n_in + (n_obj * case["n_f"] * el if power else 0) + 40 * n_obj * case["top_k"], "flops": flops}


# ---------------------------------------------------------- in plain 64 bits
def _sums(tau, weights, f_min, df, n_f):
    """[sum_j w_j exp(2 pi i f_k tau_j) for w in weights] and sum_j wl_j exp(4 pi i f_k tau_j), wl the last
    weight, for every k: a product of two phase tables, k = k1 * r + k2."""
    r = int(math.ceil(math.sqrt(n_f)))
    q = (n_f + r - 1) // r
    at = 2 * math.pi * torch.frac((f_min + df * r * torch.arange(q, device=DEV, dtype=torch.float64))[:, None] * tau)
    bt = 2 * math.pi * torch.frac((df * torch.arange(r, device=DEV, dtype=torch.float64))[:, None] * tau)
    a, b = torch.polar(torch.ones_like(at), at), torch.polar(torch.ones_like(bt), bt).T.contiguous()
    out = [((a * w) @ b).reshape(-1)[:n_f] for w in weights]
    return out + [((a * a * weights[-1]) @ (b * b)).reshape(-1)[:n_f]]


def _exact_powers(case, t, y, dy):
    """The periodogram of one object in 64 bits."""
    df = (case["f_max"] - case["f_min"]) / case["n_f"]
    n = t.numel()
    tau = t - 0.5 * (t.min() + t.max())
    if case["kind"] == "gls":
        w = 1.0 / dy ** 2
        ws = w.sum()
        yc = y - (w * y).sum() / ws
        u = w * yc
        weights = [u, w]
    else:
        yc = y - y.mean()
        weights = [yc, torch.ones_like(yc)]
    acc = None
    for i in range(0, n, 16384):
        part = _sums(tau[i:i + 16384], [v[i:i + 16384] for v in weights], case["f_min"], df, case["n_f"])
        acc = part if acc is None else [p + q for p, q in zip(acc, part)]
    z, c1, w2 = acc
    if case["kind"] == "gls":
        yy = (u * yc).sum()
        cc = 0.5 * (ws + w2.real) - c1.real ** 2 / ws
        ss = 0.5 * (ws - w2.real) - c1.imag ** 2 / ws
        cs = 0.5 * w2.imag - c1.real * c1.imag / ws
        p = (ss * z.real ** 2 + cc * z.imag ** 2 - 2 * cs * z.real * z.imag) / (yy * (cc * ss - cs * cs))
        return p if case["norm"] == "standard" else 0.5 * yy * p
    rr = w2.abs()
    z2 = z.abs() ** 2
    qq = torch.where(rr > 0, (z * z * w2.conj()).real / rr, torch.zeros_like(rr))
    d1, d2 = n + rr, n - rr
    zero = torch.zeros_like(rr)
    p = 0.5 * ((z2 + qq).clamp_min(0) / d1 + torch.where(d2 > 2e-12 * n, (z2 - qq).clamp_min(0) / d2, zero))
    return p if case["norm"] == "psd" else 2 * p / (yc * yc).sum()


def _exact_peaks(p, k):
    """The first maximum, or the k largest local maxima, on the device: (powers, bins)."""
    if k == 1:
        i = torch.argmax(p)
        return p[i][None], i[None]
    low = torch.full((1,), -math.inf, device=p.device, dtype=p.dtype)
    left, right = torch.cat([low, p[:-1]]), torch.cat([p[1:], low])
    return torch.topk(torch.where((p > left) & (p >= right), p, low), k)


def _exact_train(case, seed):
    """Loss, gradients and the first AdamW step in 64 bits, from the 16-bit weights and inputs."""
    s = prepare(case, seed)
    net = s["net"]
    widths = [learned.FEAT_DIM] + [net.dims.hidden] * net.dims.n_hidden + [net.dims.n_classes]
    p32, p16 = net.params.double(), net.params16.double()
    ws, at = [], 0
    for i, o in zip(widths[:-1], widths[1:]):
        ws.append((p16[at:at + i * o].reshape(i, o), p32[at + i * o:at + i * o + o]))
        at += i * o + o
    hs = [s["x"].double()]
    for li, (w, b) in enumerate(ws):
        z = hs[-1] @ w + b
        hs.append(z.clamp_min(0) if li + 1 < len(ws) else z)
    lab = s["labels"].long()
    loss = torch.nn.functional.cross_entropy(hs[-1], lab)
    d = torch.softmax(hs[-1], 1)
    d[torch.arange(len(lab), device=DEV), lab] -= 1
    d /= len(lab)
    grads = []
    for li in range(len(ws) - 1, -1, -1):
        grads = [(hs[li].T @ d).reshape(-1), d.sum(0)] + grads
        if li:
            d = (d @ ws[li][0].T) * (hs[li] > 0)
    g = torch.cat(grads)
    step = g / (g.abs() + 1e-8) + 1e-4 * p32
    return {"loss": loss.reshape(1), "grad": g, "params": p32 - 1e-3 * step, "m": 0.1 * g, "v": 0.001 * g * g}


def exact(case, seed):
    if case["kind"] == "learned":
        return None  # which windows are looked at is the network's choice
    if case["kind"] == "train":
        return _exact_train(case, seed)
    t, y, dy, off = _light_curves(case, seed)
    y, dy, ends = y.double(), dy.double(), off.tolist()
    want_power = case["kind"] == "single" or case.get("power", False)
    pw, ix, rows = [], [], []
    for a, b in zip(ends[:-1], ends[1:]):
        p = _exact_powers(case, t[a:b], y[a:b], dy[a:b])
        v, i = _exact_peaks(p, case["top_k"])
        pw.append(v)
        ix.append(i)
        if want_power:
            rows.append(p)
    freq = case["f_min"] + torch.stack(ix).double() * ((case["f_max"] - case["f_min"]) / case["n_f"])
    out = {"idx": None, "peak_power": torch.stack(pw), "freq_period": torch.stack([freq, 1.0 / freq], -1),
           "flags": None}
    if want_power:
        out["power"] = rows[0] if case["kind"] == "single" else torch.stack(rows)
    return out
