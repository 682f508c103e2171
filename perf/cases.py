"""The workloads that the library is timed on, through its public entry points.

A case is a dict of plain values; ``kind`` says which call it stands for:

* ``score``  one group of files classified with a count model (``score``);
* ``batch``  many groups of uneven size in one call (``Batch.score``);
* ``gw``     the group-wise method over full opcode histograms (``Groupwise.classify``);
* ``fit``    re-training a resident count model (``refit``) and reading its parameters;
* ``gauss``  re-training a resident Gaussian model, classifying a group with it, and
  reading its parameters.

Inputs are synthetic, made on the GPU from the seed: class profiles ~ Dirichlet, file totals
~ round(lognormal(8.5, 1)), counts ~ Poisson, labels Bernoulli(0.5) (two classes) or Zipf(1.1)
(families); Gaussian features around class means U(0, 10) with deviations U(0.5, 3).
"""
import math

import numpy as np
import torch

import paper_1905_13746_gb300 as nb

DEV = "cuda"
CHUNK = 1 << 28               # values generated, or computed in 64 bits, at a time
BINS, BIN_BYTES, MIN_FILES = 100, 5 * 1024, 6


def listed():
    return [
        # one arriving group of median size, in the serving configuration: latency
        {"name": "score_group", "kind": "score", "C": 2, "F": 2048, "n": 500, "dtype": "u8",
         "logpost": True},
        # the benchmark's scoring call: 16-bit counts stored as bytes and an overflow list
        {"name": "score_u8_overflow", "kind": "score", "C": 2, "F": 1024, "n": 1_000_000,
         "dtype": "u8ovf", "logpost": True},
        # a wide vocabulary in the smallest exact float format
        {"name": "score_fp8_wide", "kind": "score", "C": 2, "F": 4096, "n": 250_007,
         "dtype": "fp8", "logpost": True},
        # plain float counts just as a user's tensor holds them: odd width, labels only
        {"name": "score_f32_odd", "kind": "score", "C": 2, "F": 1003, "n": 100_003,
         "dtype": "f32", "logpost": False},
        # family classification: 64 families over the full opcode n-gram table
        {"name": "score_families", "kind": "score", "C": 64, "F": 8192, "n": 262_144,
         "dtype": "u8", "logpost": True},
        # family classification with 16 families from BF16 counts, ragged group
        {"name": "score_families_bf16", "kind": "score", "C": 16, "F": 2048, "n": 150_001,
         "dtype": "bf16", "logpost": True},
        # one step of the serving loop: groups of two models scored together
        {"name": "batch_step", "kind": "batch", "F": 2048, "groups": 64, "median": 500,
         "logpost": True},
        # the paper's method at its largest selection: 100 size groups, 200 opcodes each
        {"name": "groupwise", "kind": "gw", "F": 1024, "n": 500_000, "k": 200},
        # the benchmark's re-training call
        {"name": "fit_u8_overflow", "kind": "fit", "C": 2, "F": 1024, "n": 666_667,
         "dtype": "u8ovf"},
        # re-training the family model
        {"name": "fit_families", "kind": "fit", "C": 64, "F": 8192, "n": 262_144, "dtype": "u8"},
        # real-valued features, the small workload: 1,000 training files per class
        {"name": "gauss_small", "kind": "gauss", "C": 2, "F": 64, "n_fit": 2000, "n": 10_000,
         "logpost": True},
        # real-valued features, 64 families
        {"name": "gauss_families", "kind": "gauss", "C": 64, "F": 256, "n_fit": 64_000,
         "n": 200_000, "logpost": True},
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["score", "score", "score", "batch", "gw", "fit", "fit", "gauss", "gauss"])
    if kind == "score":
        dtype = rng.choice(["u8", "u8ovf", "fp8", "bf16", "f32"])
        C = 2 if dtype in ("u8ovf", "f32") else rng.choice([2, 2, rng.randint(3, 64)])
        # up to 2 GB of rows for bytes, 1 GB for the wider types and the two-class models; the
        # families are bounded by their products too
        F = _log(rng, 64, 8192)
        size = {"f32": 4, "bf16": 2}.get(dtype, 1)
        most = 1e9 / (size * F) if C == 2 else min(1e9 / (size * F), 1.2e11 / (C * F))
        if dtype == "f32":
            most = min(most, 1e8 / F)
        return {"kind": kind, "C": C, "F": F, "n": _log(rng, 100, max(200, int(most))),
                "dtype": dtype, "logpost": rng.random() < 0.75}
    if kind == "batch":
        return {"kind": kind, "F": rng.choice([256, 512, 1024, 2048, 2000]),
                "groups": rng.randint(8, 128), "median": _log(rng, 50, 1000),
                "logpost": rng.random() < 0.75}
    if kind == "gw":
        return {"kind": kind, "F": rng.choice([512, 1000, 1024, 2048]),
                "n": _log(rng, 5000, 400_000), "k": rng.choice([20, 40, 80, 100, 160, 200])}
    if kind == "fit":
        dtype = rng.choice(["u8", "u8", "u8ovf", "fp8", "bf16", "f32"])
        C = 2 if dtype == "u8ovf" else rng.choice([2, rng.randint(3, 64)])
        F = _log(rng, 64, 8192)
        size = {"f32": 4, "bf16": 2}.get(dtype, 1)
        return {"kind": kind, "C": C, "F": F, "dtype": dtype,
                "n": _log(rng, 2000, max(4000, int(6e8 / (size * F))))}
    C = rng.choice([2, rng.randint(3, 64)])
    F = _log(rng, 16, 512)
    return {"kind": kind, "C": C, "F": F, "n_fit": _log(rng, 20 * C, int(1.2e7 / F)),
            "n": _log(rng, 1000, int(min(5e7 / F, 3e9 / (C * F)))),
            "logpost": rng.random() < 0.75}


# ---- inputs ----------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _profiles(rng, shape, conc):
    g = np.maximum(rng.standard_gamma(conc, size=shape), 1e-30)
    return torch.from_numpy((g / g.sum(-1, keepdims=True)).astype(np.float32)).to(DEV)


def _labels(g, n, C, every=False):
    """Bernoulli(0.5) for two classes, Zipf(1.1) for more; `every`: no class without files."""
    w = torch.ones(2, device=DEV) if C == 2 else \
        (torch.arange(C, device=DEV, dtype=torch.float32) + 1.0) ** -1.1
    edges = (w / w.sum()).cumsum(0)
    y = torch.bucketize(torch.rand(n, generator=g, device=DEV), edges[:-1].contiguous())
    if every:
        y[:C] = torch.arange(C, device=DEV)
    return y.to(torch.int32)


def _counts(g, p, row, total, clip, dtype, ld=None):
    """Poisson(total_i p[row_i, :]) clipped, n x F (a view of n x ld where ld is given)."""
    n, F = row.shape[0], p.shape[1]
    out = (torch.zeros if ld else torch.empty)((n, ld or F), dtype=dtype, device=DEV)
    step = max(1, CHUNK // F)
    for a in range(0, n, step):
        r = p[row[a:a + step].long()]
        r *= total[a:a + step, None]
        x = torch.poisson(r, generator=g).clamp_(max=clip)
        out[a:a + step, :F] = x.to(torch.int32).to(dtype) if dtype == torch.uint16 else x.to(dtype)
    return out[:, :F]


def _totals(g, n):
    return torch.exp(8.5 + torch.randn(n, generator=g, device=DEV)).round_()


def _raw(g, p, y, dtype):
    """The files' counts as the storage format holds them exactly, before packing."""
    F, total = p.shape[1], _totals(g, y.shape[0])
    if dtype == "u8ovf":
        return _counts(g, p, y, total, 65535, torch.uint16)
    if dtype == "f32":
        return _counts(g, p, y, total, 65535, torch.float32)
    if dtype == "bf16":
        return _counts(g, p, y, total, 255, torch.bfloat16, (F + 7) // 8 * 8)
    return _counts(g, p, y, total, 255, torch.uint8, (F + 15) // 16 * 16)


def _stored(x, dtype):
    if dtype == "u8ovf":
        return nb.pack_u8(x)
    if dtype == "fp8":
        return nb.pack_fp8(x.to(torch.float32))
    return nb.Features(x)


def _stored64(x, dtype):
    """The values that the stored form of x stands for, in 64 bits."""
    if dtype == "u8ovf":
        return x.to(torch.int32).double()
    x = x.float()
    if dtype == "fp8":         # 255 is below 448: no row is scaled
        x = x.to(torch.float8_e4m3fn).float()
    return x.double()


def _count_inputs(case, seed, fit_rows, score_rows):
    rng, g = np.random.default_rng(seed), _gen(seed)
    C, F, dtype = case["C"], case["F"], case["dtype"]
    p = _profiles(rng, (C, F), 0.1)
    y = _labels(g, fit_rows, C, every=True)
    x = _raw(g, p, y, dtype)
    z = _raw(g, p, _labels(g, score_rows, C), dtype) if score_rows else None
    return x, y, z


def _fit_rows(case):
    """Training files behind a scoring case's model: enough for every family."""
    return 16_384 if case["C"] == 2 else 32_768


def _gauss_inputs(case, seed):
    rng, g = np.random.default_rng(seed), _gen(seed)
    C, F = case["C"], case["F"]
    mu = torch.from_numpy(rng.uniform(0.0, 10.0, (C, F)).astype(np.float32)).to(DEV)
    sd = torch.from_numpy(rng.uniform(0.5, 3.0, (C, F)).astype(np.float32)).to(DEV)

    def files(n, every):
        y = torch.randint(C, (n,), generator=g, device=DEV)
        if every:
            y[:2 * C] = torch.arange(2 * C, device=DEV) % C
        x = torch.randn((n, F), generator=g, device=DEV).mul_(sd[y]).add_(mu[y])
        return x, y.to(torch.int32)

    x, y = files(case["n_fit"], True)
    return x, y, files(case["n"], False)[0]


def _batch_inputs(case, seed):
    """Two models (2 and 16 families) and the groups of one step."""
    rng, g = np.random.default_rng(seed), _gen(seed)
    F, models = case["F"], []
    for C in (2, 16):
        p = _profiles(rng, (C, F), 0.05)
        y = _labels(g, 16_384, C, every=True)
        models.append((C, p, _counts(g, p, y, _totals(g, 16_384), 255, torch.uint8), y))
    # sizes from the case alone, so that passes over other inputs do the same work
    size = np.random.default_rng(case["groups"] * 131 + case["median"])
    n = np.clip(np.rint(size.lognormal(math.log(case["median"]), 1.49, case["groups"])),
                1, 50_000).astype(np.int64)
    slot = np.arange(case["groups"]) % 2
    groups = []
    for k in range(2):
        _, p = models[k][:2]
        m = int(n[slot == k].sum())
        groups.append(_counts(g, p, _labels(g, m, models[k][0]), _totals(g, m), 255, torch.uint8,
                              (F + 15) // 16 * 16))
    return models, n, slot, groups


def _gw_inputs(case, seed):
    rng, g = np.random.default_rng(seed), _gen(seed)
    n_fit, F = 150_000, case["F"]
    n = n_fit + case["n"]
    at = np.arange(BINS) + 0.5
    w = np.exp(-0.5 * np.log(at / 12.0) ** 2) / at
    edges = torch.from_numpy((w / w.sum()).cumsum()[:-1].astype(np.float32)).to(DEV)
    win = torch.bucketize(torch.rand(n, generator=g, device=DEV), edges)
    size = win * BIN_BYTES + torch.randint(BIN_BYTES, (n,), generator=g, device=DEV)
    y = (torch.rand(n, generator=g, device=DEV) < 0.827).to(torch.int32)
    p = 0.5 * _profiles(rng, (2, F), 0.1)[None] + 0.5 * _profiles(rng, (BINS, 2, F), 0.1)
    total = (size // 16).clamp_(min=1).float()
    x = _counts(g, p.reshape(2 * BINS, F), win * 2 + y, total, 255, torch.uint8,
                (F + 15) // 16 * 16)
    return x[:n_fit], y[:n_fit], size[:n_fit].contiguous(), x[n_fit:], size[n_fit:].contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "score":
        x, y, z = _count_inputs(case, seed, _fit_rows(case), case["n"])
        model = nb.fit(_stored(x, case["dtype"]), y, case["C"])
        return {"case": case, "model": model, "X": _stored(z, case["dtype"])}
    if kind == "fit":
        x, y, _ = _count_inputs(case, seed, case["n"], 0)
        X = _stored(x, case["dtype"])
        return {"case": case, "X": X, "y": y, "model": nb.fit(X, y, case["C"])}
    if kind == "gauss":
        x, y, z = _gauss_inputs(case, seed)
        model = nb.fit(x, y, case["C"], kind=nb.NB_GAUSSIAN)
        return {"case": case, "model": model, "X": x, "y": y, "Z": z}
    if kind == "gw":
        x, y, size, z, zsize = _gw_inputs(case, seed)
        t = nb.fit_groupwise(x, y, size, case["k"])
        gw = nb.Groupwise(t["models"], t["cols"], t["model_of"], case["F"], max_files=case["n"])
        return {"case": case, "gw": gw, "X": z, "size": zsize}
    models, n, slot, rows = _batch_inputs(case, seed)
    fitted = [nb.fit(x, y, C) for C, _, x, y in models]
    batch = nb.Batch(fitted, nb.NB_U8, rows[0].stride(0), case["groups"],
                     want_logpost=case["logpost"])
    out = [batch.outputs(k, rows[k].shape[0]) for k in range(2)]
    groups, at = [], [0, 0]
    for k, m in zip(slot.tolist(), n.tolist()):
        a, b = at[k], at[k] + m
        part = {name: t[a:b] if t is not None else None for name, t in out[k].items()}
        groups.append((k, nb.Features(rows[k][a:b]), part))
        at[k] = b
    return {"case": case, "batch": batch, "groups": groups, "out": out}


def _result(r):
    return {name: r[name] for name in ("label", "margin", "logpost")}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "score":
        return _result(nb.score(state["model"], state["X"], want_logpost=case["logpost"]))
    if kind == "fit":
        m = nb.refit(state["model"], state["X"], state["y"])
        p0, _, log_pi = m.params()
        return {"log_theta": p0, "log_pi": log_pi}
    if kind == "gauss":
        m = nb.refit(state["model"], state["X"], state["y"], no_sync=True)
        r = _result(nb.score(m, state["Z"], want_logpost=case["logpost"]))
        mu, var, log_pi = m.params()
        return dict(r, mu=mu, var=var, log_pi=log_pi)
    if kind == "gw":
        return _result(state["gw"].classify(state["X"], state["size"]))
    state["batch"].score(state["groups"])
    return [_result(r) for r in state["out"]]


# ---- what one pass cannot do without ----------------------------------------
def _out_bytes(n, C, logpost):
    return n * (5 + (4 * C if logpost else 0))


def _row_bytes(case):
    F = case["F"]
    return {"u8": F, "u8ovf": F + 8, "fp8": F + 1, "bf16": 2 * F, "f32": 4 * F}[case["dtype"]]


def work(case):
    kind, F = case["kind"], case["F"]
    if kind == "score":
        C, n = case["C"], case["n"]
        return {"bytes": n * _row_bytes(case) + 8 * C * F + _out_bytes(n, C, case["logpost"]),
                "flops": 2.0 * n * F * (C if C > 2 else 1)}
    if kind == "fit":
        return {"bytes": case["n"] * (_row_bytes(case) + 4) + 8 * case["C"] * F,
                "flops": 1.0 * case["n"] * F}
    if kind == "gauss":
        C, n = case["C"], case["n"]
        return {"bytes": 4 * F * (case["n_fit"] + n) + 4 * case["n_fit"] + 16 * C * F
                + _out_bytes(n, C, case["logpost"]),
                "flops": 3.0 * F * (case["n_fit"] + C * n)}
    if kind == "gw":
        return {"bytes": case["n"] * (F + 8) + _out_bytes(case["n"], 2, True),
                "flops": 2.0 * case["n"] * case["k"]}
    size = np.random.default_rng(case["groups"] * 131 + case["median"])
    n = np.clip(np.rint(size.lognormal(math.log(case["median"]), 1.49, case["groups"])), 1, 50_000)
    two, many = float(n[0::2].sum()), float(n[1::2].sum())
    return {"bytes": (two + many) * F + _out_bytes(two, 2, case["logpost"])
            + _out_bytes(many, 16, case["logpost"]), "flops": 2.0 * F * (two + 16 * many)}


# ---- the same in 64 bits ------------------------------------------------------
def _fit64(x, y, C, dtype):
    """log theta (C x F) and log pi of the multinomial model, alpha = 1."""
    n, F = x.shape
    counts = torch.zeros((C, F), dtype=torch.float64, device=DEV)
    step = max(1, CHUNK // (4 * F))
    for a in range(0, n, step):
        hot = torch.nn.functional.one_hot(y[a:a + step].long(), C).double()
        counts += hot.T @ _stored64(x[a:a + step], dtype)
    log_theta = (counts + 1.0).log() - (counts.sum(1, keepdim=True) + F).log()
    nc = torch.bincount(y.long(), minlength=C).double()
    return log_theta, nc.log() - math.log(n)


def _decide64(s, logpost):
    top = s.topk(2, dim=1).values
    return {"label": s.argmax(1).to(torch.uint8), "margin": top[:, 0] - top[:, 1],
            "logpost": torch.log_softmax(s, 1) if logpost else None}


def _joined(parts):
    return {k: None if parts[0][k] is None else torch.cat([r[k] for r in parts])
            for k in parts[0]}


def _score64(x, log_theta, log_pi, dtype, logpost):
    step = max(1, CHUNK // (4 * x.shape[1]))
    return _joined([_decide64(_stored64(x[a:a + step], dtype) @ log_theta.T + log_pi, logpost)
                    for a in range(0, x.shape[0], step)])


def _gauss64(case, seed):
    x, y, z = _gauss_inputs(case, seed)
    C, F, n = case["C"], case["F"], x.shape[0]
    x64, lab = x.double(), y.long()
    nc = torch.bincount(lab, minlength=C).double()
    mu = torch.stack([x64[lab == c].mean(0) for c in range(C)])
    var = torch.stack([(x64[lab == c] - mu[c]).square().mean(0) for c in range(C)])
    var += 1e-9 * (x64 - x64.mean(0)).square().mean(0).max()
    log_pi = nc.log() - math.log(n)
    const = log_pi - 0.5 * (2.0 * math.pi * var).log().sum(1)
    parts, step = [], max(1, CHUNK // (8 * F))
    for a in range(0, z.shape[0], step):
        b = z[a:a + step].double()
        s = torch.stack([const[c] - 0.5 * ((b - mu[c]).square() / var[c]).sum(1)
                         for c in range(C)], 1)
        parts.append(_decide64(s, case["logpost"]))
    return dict(_joined(parts), mu=mu, var=var, log_pi=log_pi)


def _gw64(case, seed):
    """The per-group models (Laplace, on each group's top k opcodes) and their scores."""
    x, y, size, z, zsize = _gw_inputs(case, seed)
    k, F = case["k"], case["F"]
    win, zwin = size // BIN_BYTES, zsize // BIN_BYTES
    per = torch.bincount(win * 2 + y, minlength=2 * BINS).reshape(BINS, 2).cpu()
    trained = [w for w in range(BINS) if int(per[w].min()) >= MIN_FILES]
    label = torch.zeros(z.shape[0], dtype=torch.uint8, device=DEV)
    margin = torch.zeros(z.shape[0], dtype=torch.float64, device=DEV)
    logpost = torch.zeros((z.shape[0], 2), dtype=torch.float64, device=DEV)
    fitted = {}
    for w in range(BINS):
        of = next((t for t in trained if t >= w), trained[-1])
        if of not in fitted:
            rows = (win == of).nonzero()[:, 0]
            xs, ys = x[rows], y[rows]
            N = torch.stack([xs[ys == c].sum(0, dtype=torch.int64) for c in range(2)])
            D = N.sum(1)
            key = (N[1] * D[0] - N[0] * D[1]).abs()
            cols = torch.sort(key, descending=True, stable=True).indices[:k]
            fitted[of] = (cols, *_fit64(xs[:, cols], ys, 2, "u8"))
        cols, log_theta, log_pi = fitted[of]
        at = (zwin == w).nonzero()[:, 0]
        if not at.numel():
            continue
        r = _score64(z[at][:, cols], log_theta, log_pi, "u8", True)
        label[at], margin[at], logpost[at] = r["label"], r["margin"], r["logpost"]
    return {"label": label, "margin": margin, "logpost": logpost}


def exact(case, seed):
    kind = case["kind"]
    if kind == "score":
        x, y, z = _count_inputs(case, seed, _fit_rows(case), case["n"])
        log_theta, log_pi = _fit64(x, y, case["C"], case["dtype"])
        return _score64(z, log_theta, log_pi, case["dtype"], case["logpost"])
    if kind == "fit":
        x, y, _ = _count_inputs(case, seed, case["n"], 0)
        log_theta, log_pi = _fit64(x, y, case["C"], case["dtype"])
        return {"log_theta": log_theta, "log_pi": log_pi}
    if kind == "gauss":
        return _gauss64(case, seed)
    if kind == "gw":
        return _gw64(case, seed)
    models, _, _, rows = _batch_inputs(case, seed)
    return [_score64(rows[k], *_fit64(models[k][2], models[k][3], models[k][0], "u8"), "u8",
                     case["logpost"]) for k in range(2)]
