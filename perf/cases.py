"""The work that callers of this library have it do, as measurable cases.

A pass is the scoring of one batch through the binding, as a serving loop does it: a fresh segment
plan for the batch's offsets, then the layers that share it.  Weights, output buffers and workspaces
live as long as the program and are made once; inputs are N(0, 1) and weights N(0, 1 / fan_in), the
distributions of the repository's own workloads.  Segment sizes follow the four laws those workloads
name (constant, uniform, log-normal, Zipf) and belong to the case, not to the seed of the inputs.

Kinds of batch:
  mlp    retrieval tower: split layer (request half broadcast in the kernel) and two plain layers
  norm   the same tower with group-local normalisation: inputs normalised per group, the middle
         normalisation folded into the layers around it
  dca    ranking: query projection of the candidates, then cross attention over the request's sequence
  glm    pairwise interaction under the isolation mask, raw block and / or row-axis compression
  fm     pairwise interaction projected to k columns
  block  mixed block: split layer, cross attention and interaction on one plan
"""
import math

import numpy as np
import torch

from paper_2607_27744_b200 import binding as rocs

BF16, F32 = "bf16", "f32"
_DTYPE = {BF16: torch.bfloat16, F32: torch.float32}
_SIZE = {BF16: 2, F32: 4}


def listed():
    return [
        # The smallest block anybody scores, in fp32: 4 requests with 1..16 candidates each, every
        # operator once.  Nothing here is large; launches and host work are the time.
        {"name": "tiny_f32_block", "kind": "block", "dtype": F32, "R": 4, "law": "uniform", "per": 8, "segments": 1,
         "d_req": 64, "d_cand": 32, "d_out": 64, "relu": False, "H": 2, "dh": 32, "L_lo": 32, "L_hi": 32,
         "n_r": 4, "n_c": 2, "d": 16, "n_ro": 0, "n_co": 0},
        # The fp32 path at the widths of the mixed block, for callers that do not round to bf16: a
        # handful of requests with about a hundred candidates each and short histories.
        {"name": "f32_block", "kind": "block", "dtype": F32, "R": 24, "law": "lognormal", "per": 110, "segments": 2,
         "d_req": 768, "d_cand": 256, "d_out": 1024, "relu": True, "H": 8, "dh": 64, "L_lo": 64, "L_hi": 384,
         "n_r": 24, "n_c": 8, "d": 128, "n_ro": 4, "n_co": 4},
        # Online retrieval: one request, a few hundred candidates, the tower's full widths.
        {"name": "online_retrieval", "kind": "mlp", "dtype": BF16, "R": 1, "law": "const", "per": 500, "segments": 3,
         "d_req": 512, "d_cand": 256, "hidden": 1024, "middle": 1024, "d_out": 256, "bias": True},
        # A micro-batch of requests collected over a few milliseconds, ragged.
        {"name": "microbatch_retrieval", "kind": "mlp", "dtype": BF16, "R": 12, "law": "lognormal", "per": 400,
         "segments": 4, "d_req": 512, "d_cand": 256, "hidden": 1024, "middle": 1024, "d_out": 256, "bias": True},
        # Bulk retrieval: 256 requests x 512 candidates, the repository's headline workload.
        {"name": "bulk_retrieval", "kind": "mlp", "dtype": BF16, "R": 256, "law": "const", "per": 512, "segments": 5,
         "d_req": 512, "d_cand": 256, "hidden": 1024, "middle": 1024, "d_out": 256, "bias": False},
        # The normalised tower on a ragged batch.
        {"name": "normed_tower", "kind": "norm", "dtype": BF16, "R": 96, "law": "lognormal", "per": 450, "segments": 6,
         "d_req": 512, "d_cand": 256, "hidden": 1024, "d_out": 512, "norm": "rms"},
        # Online ranking: a few requests with long histories, too few query tiles to fill the chip.
        {"name": "online_ranking", "kind": "dca", "dtype": BF16, "R": 3, "law": "lognormal", "per": 250, "segments": 7,
         "d_feat": 512, "H": 8, "dh": 64, "n_q": 1, "L_lo": 1000, "L_hi": 2048},
        # Bulk ranking: 64 requests, log-normal candidates, 2048 tokens, 8 heads of 64.
        {"name": "bulk_ranking", "kind": "dca", "dtype": BF16, "R": 64, "law": "lognormal", "per": 900, "segments": 8,
         "d_feat": 512, "H": 8, "dh": 64, "n_q": 1, "L_lo": 2048, "L_hi": 2048},
        # Several query tokens per candidate on wide heads, ragged sequences.
        {"name": "token_ranking", "kind": "dca", "dtype": BF16, "R": 40, "law": "lognormal", "per": 24, "segments": 9,
         "d_feat": 256, "H": 4, "dh": 128, "n_q": 32, "L_lo": 500, "L_hi": 1500},
        # Interaction with compression: 128 requests x 1024 candidates, 32 + 16 embeddings of 128.
        {"name": "bulk_interaction", "kind": "glm", "dtype": BF16, "R": 128, "law": "const", "per": 1024, "segments": 10,
         "n_r": 32, "n_c": 16, "d": 128, "n_ro": 8, "n_co": 8, "raw": False},
        # Projected interaction of a ragged batch with embedding counts that are no powers of two.
        {"name": "ragged_projection", "kind": "fm", "dtype": BF16, "R": 100, "law": "lognormal", "per": 200, "segments": 11,
         "n_r": 20, "n_c": 12, "d": 128, "k": 16},
        # The heaviest batch: 1024 requests with Zipf candidates (about 1.5 million), every operator.
        {"name": "skewed_block", "kind": "block", "dtype": BF16, "R": 1024, "law": "zipf", "per": 8192, "segments": 12,
         "d_req": 768, "d_cand": 256, "d_out": 1024, "relu": False, "H": 8, "dh": 64, "L_lo": 256, "L_hi": 1024,
         "n_r": 24, "n_c": 8, "d": 128, "n_ro": 0, "n_co": 0},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["mlp", "mlp", "norm", "dca", "dca", "glm", "fm", "block", "block"])
    case = {"kind": kind, "dtype": BF16, "segments": rng.randrange(100, 1 << 20)}

    def requests(most_candidates, least=1):
        n = log_int(max(least, 8), most_candidates)
        case["R"] = log_int(1, min(256, max(1, n // 8)))
        case["law"] = rng.choice(["const", "uniform", "lognormal"])
        case["per"] = max(1, -(-n // case["R"]))

    if kind in ("mlp", "norm"):
        requests(120000, 6000 if kind == "norm" else 1)   # the folded normalisation starts at 2048 rows
        case.update(d_req=8 * log_int(16, 96), d_cand=rng.choice([64, 128, 200, 256, 256, 384, 512]),
                    hidden=rng.choice([512, 768, 1024, 1024]), d_out=rng.choice([256, 320, 512]))
        if kind == "mlp":
            case.update(middle=rng.choice([256, 512, 1000, 1024]), bias=rng.random() < 0.5)
        else:
            case["norm"] = rng.choice(["rms", "layer"])
    elif kind == "dca":
        dh = rng.choice([32, 64, 64, 128])
        n_q = rng.choice([1, 1, 1, 5, 32])
        requests(50000 // n_q)
        L = log_int(40, 2048)
        case.update(d_feat=rng.choice([256, 512]), H=max(1, rng.choice([256, 512]) // dh), dh=dh, n_q=n_q,
                    L_lo=max(1, L // 2), L_hi=L)
    elif kind in ("glm", "fm"):
        requests(60000)
        case.update(n_r=rng.choice([8, 16, 20, 24, 32, 48]), n_c=rng.choice([4, 8, 12, 16, 16]),
                    d=rng.choice([64, 128, 128, 192]))
        if kind == "fm":
            case["k"] = rng.choice([8, 16, 16, 24])
        else:
            n_ro = rng.choice([0, 4, 8])
            case.update(n_ro=n_ro, n_co=n_ro, raw=n_ro == 0 or rng.random() < 0.3)
    else:
        f32 = rng.random() < 0.5
        requests(3000 if f32 else 40000)
        case["dtype"] = F32 if f32 else BF16
        dh = rng.choice([32, 64]) if f32 else rng.choice([32, 64, 128])
        L = log_int(32, 400 if f32 else 1024)
        n_ro = rng.choice([0, 4, 8])
        case.update(d_req=8 * log_int(8, 96), d_cand=rng.choice([32, 64, 128, 200, 256]), relu=rng.random() < 0.5,
                    d_out=rng.choice([64, 256, 512, 1024]), H=max(1, rng.choice([128, 512]) // dh), dh=dh,
                    L_lo=max(1, L // 2), L_hi=L, n_r=rng.choice([4, 8, 24, 32]), n_c=rng.choice([2, 8, 16]),
                    d=rng.choice([16, 64, 128]), n_ro=n_ro, n_co=n_ro)
    return case


# ---------------------------------------------------------------------------------- segments
def _counts(case):
    """Candidates of each request."""
    g, R, per = np.random.default_rng([2607, case["segments"]]), case["R"], case["per"]
    if case["law"] == "const":
        return np.full(R, per, np.int64)
    if case["law"] == "uniform":
        return g.integers(1, 2 * per + 1, size=R)
    if case["law"] == "lognormal":                       # mean about `per`, the tail cut at eight times that
        return np.clip(np.rint(g.lognormal(math.log(per) - 0.32, 0.8, size=R)), 1, 8 * per).astype(np.int64)
    return np.clip(g.zipf(1.2, size=R), 1, per).astype(np.int64)


def _lengths(case):
    """Sequence positions of each request."""
    return np.random.default_rng([2608, case["segments"]]).integers(case["L_lo"], case["L_hi"] + 1, size=case["R"])


def _rows(case):
    """Candidates of the batch; the normalised tower pads its batch to the fold's smallest row count."""
    n = int(_counts(case).sum())
    return max(n, 2048) if case["kind"] == "norm" else n


def _offsets(case):
    counts = _counts(case)
    counts[-1] += _rows(case) - int(counts.sum())
    return np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)


# ---------------------------------------------------------------------------------- inputs
def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dt, kind, R, N = _DTYPE[case["dtype"]], case["kind"], case["R"], _rows(case)
    off = _offsets(case)

    def normal(*shape, std=1.0, dtype=dt):
        t = torch.empty(shape, dtype=dtype, device="cuda").normal_(generator=gen)
        return t if std == 1.0 else t.mul_(std)

    def empty(*shape, dtype=dt):
        return torch.empty(shape, dtype=dtype, device="cuda")

    s = {"case": case, "offsets_host": torch.from_numpy(off), "offsets": torch.from_numpy(off).cuda()}
    plan = rocs.plan_create(s["offsets"], s["offsets_host"])     # only to size the workspaces

    if kind in ("mlp", "norm", "block"):
        d_req, d_cand = case["d_req"], case["d_cand"]
        d_first = case["d_out"] if kind == "block" else case["hidden"]
        W = normal(d_first, d_req + d_cand, std=(d_req + d_cand) ** -0.5)
        s.update(XR=normal(R, d_req), XC=normal(N, d_cand), W_CR=W[:, :d_req], W_CC=W[:, d_req:], y1=empty(N, d_first))
        if kind == "norm":
            need = int(rocs.lib().rocs_ikbo_linear_stats_workspace(plan.handle, d_first))
        else:
            need = rocs.ikbo_linear_workspace(plan, d_first)
        s["ws1"] = empty(need, dtype=torch.uint8)
    if kind == "mlp":
        hidden, middle, d_out = case["hidden"], case["middle"], case["d_out"]
        s.update(W2=normal(middle, hidden, std=hidden ** -0.5), W3=normal(d_out, middle, std=middle ** -0.5),
                 y2=empty(N, middle), y3=empty(N, d_out), b1=None, b2=None, b3=None)
        if case["bias"]:
            for name, width in (("b1", hidden), ("b2", middle), ("b3", d_out)):
                s[name] = normal(width, dtype=torch.float32)
    if kind == "norm":
        hidden, d_out = case["hidden"], case["d_out"]
        gain = normal(hidden, std=0.2, dtype=torch.float32) + 1.0
        W2 = normal(d_out, hidden, std=hidden ** -0.5, dtype=torch.float32)
        s.update(W2=(W2 * gain).to(dt), b1=normal(hidden, dtype=torch.float32), b2=normal(d_out, dtype=torch.float32),
                 gR=normal(d_req, std=0.2) + 1.0, gC=normal(d_cand, std=0.2) + 1.0,
                 bR=normal(d_req, std=0.3), bC=normal(d_cand, std=0.3),
                 xr=empty(R, d_req), xc=empty(N, d_cand), stats=empty(N, 2, dtype=torch.float32), y2=empty(N, d_out))
        s["wbar"] = rocs.weight_row_sums(s["W2"])                # a weight: laid out once
    if kind in ("dca", "block"):
        lengths = _lengths(case)
        so = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
        H, dh, n_q, T = case["H"], case["dh"], case.get("n_q", 1), int(so[-1])
        s.update(seq=torch.from_numpy(so).cuda(), K=normal(T, H, dh), V=normal(T, H, dh), att=empty(N, n_q, H, dh))
        if kind == "dca":
            d_feat = case["d_feat"]
            s.update(feat=normal(N, d_feat), WQ=normal(n_q * H * dh, d_feat, std=d_feat ** -0.5),
                     Q=empty(N, n_q * H * dh))
        else:
            s["Q"] = normal(N, n_q, H, dh)
    if kind in ("glm", "fm", "block"):
        n_r, n_c, d = case["n_r"], case["n_c"], case["d"]
        n, k = n_r + n_c, case.get("k", 0)
        s.update(ER=normal(R, n_r, d), EC=normal(N, n_c, d), C=None, ws2=None, outs={})
        if kind == "fm":
            s.update(P=normal(n, k, std=n ** -0.5), ws2=empty(rocs.glm_fm_projection_workspace(plan, d, k), dtype=torch.uint8),
                     outs={"FR": empty(R, n_r, k), "FC": empty(N, n_c, k)})
        else:
            n_ro, n_co = case["n_ro"], case["n_co"]
            if n_co:
                s.update(C=normal(n_ro + n_co, n, std=n ** -0.5), ws2=empty(
                    rocs.glm_interaction_workspace(plan, n_r, n_c, n_co), dtype=torch.uint8))
                s["outs"].update(OR=empty(R, n_ro, n), OC=empty(N, n_co, n))
            if _raw(case):
                s["outs"].update(YR=empty(R, n_r, n), YC=empty(N, n_c, n))
    plan.close()
    return s


def _raw(case):
    return case.get("raw", case["n_co"] == 0)


# ---------------------------------------------------------------------------------- one pass
def run(s):
    case = s["case"]
    kind = case["kind"]
    plan = rocs.plan_create(s["offsets"], s["offsets_host"])
    if kind == "mlp":
        h = rocs.ikbo_linear(plan, s["XR"], s["XC"], s["W_CR"], s["W_CC"], bias=s["b1"], relu=True, out=s["y1"],
                             workspace=s["ws1"])
        h = rocs.linear(h, s["W2"], bias=s["b2"], relu=True, out=s["y2"])
        out = rocs.linear(h, s["W3"], bias=s["b3"], out=s["y3"])
    elif kind == "norm":
        rule = rocs.NORM_RMS if case["norm"] == "rms" else rocs.NORM_LAYER
        xr = rocs.group_norm(s["XR"], s["gR"], s["bR"], kind=rule, out=s["xr"])
        xc = rocs.group_norm(s["XC"], s["gC"], s["bC"], kind=rule, out=s["xc"])
        h, stats = rocs.ikbo_linear_stats(plan, xr, xc, s["W_CR"], s["W_CC"], bias=s["b1"], relu=True, out=s["y1"],
                                          row_stats=s["stats"], workspace=s["ws1"])
        out = rocs.linear_normed(h, stats, s["W2"], s["wbar"], bias=s["b2"], kind=rule, relu=True, out=s["y2"])
    elif kind == "dca":
        q = rocs.linear(s["feat"], s["WQ"], out=s["Q"])
        out = rocs.dca_attention(plan, q.view(s["att"].shape), s["K"], s["V"], s["seq"], out=s["att"])
    elif kind == "glm":
        out = _interaction(plan, s)
    elif kind == "fm":
        out = rocs.glm_fm_projection(plan, s["ER"], s["EC"], s["P"], workspace=s["ws2"], outs=s["outs"])
    else:
        y = rocs.ikbo_linear(plan, s["XR"], s["XC"], s["W_CR"], s["W_CC"], relu=case["relu"], out=s["y1"],
                             workspace=s["ws1"])
        a = rocs.dca_attention(plan, s["Q"], s["K"], s["V"], s["seq"], out=s["att"])
        out = {"linear": y, "attention": a, "interaction": _interaction(plan, s)}
    plan.close()
    return out


def _interaction(plan, s):
    case = s["case"]
    return rocs.glm_interaction(plan, s["ER"], s["EC"], s["C"], case["n_ro"], case["n_co"], want_raw=_raw(case),
                                workspace=s["ws2"], outs=s["outs"])


# ---------------------------------------------------------------------------------- what a pass needs
def work(case):
    kind, R, N, e = case["kind"], case["R"], _rows(case), _SIZE[case["dtype"]]
    values, flops = 0, 0                                   # values of the storage type, read or written once
    if kind in ("mlp", "norm", "block"):
        d_req, d_cand = case["d_req"], case["d_cand"]
        d_first = case["d_out"] if kind == "block" else case["hidden"]
        values += R * d_req + N * d_cand + d_first * (d_req + d_cand)
        flops += 2 * R * d_req * d_first + 2 * N * d_cand * d_first
        if kind == "block":
            values += N * d_first
        widths = [d_first] + ([case["middle"]] if kind == "mlp" else []) + ([] if kind == "block" else [case["d_out"]])
        for a, b in zip(widths, widths[1:]):
            values += a * b
            flops += 2 * N * a * b
        if kind != "block":
            values += N * widths[-1]
    if kind in ("dca", "block"):
        lengths, counts, n_q = _lengths(case), _counts(case), case.get("n_q", 1)
        width = case["H"] * case["dh"]
        values += 2 * int(lengths.sum()) * width + N * n_q * width
        flops += 4 * int((counts * lengths).sum()) * n_q * width
        if kind == "dca":
            values += N * case["d_feat"] + n_q * width * case["d_feat"]
            flops += 2 * N * n_q * width * case["d_feat"]
        else:
            values += N * n_q * width
    if kind in ("glm", "fm", "block"):
        n_r, n_c, d = case["n_r"], case["n_c"], case["d"]
        n = n_r + n_c
        values += R * n_r * d + N * n_c * d
        if kind == "fm":
            k = case["k"]
            values += n * k + R * n_r * k + N * n_c * k
            flops += 4 * R * n_r * d * k + 4 * N * n_c * d * k
        else:
            n_ro, n_co = case["n_ro"], case["n_co"]
            flops += 2 * R * n_r * n_r * d + 2 * N * n_c * n * d
            flops += 2 * R * (n_ro + n_co) * n_r * n_r + 2 * N * n_co * n_c * n
            values += (n_ro + n_co) * n + R * n_ro * n + N * n_co * n
            if _raw(case):
                values += R * n_r * n + N * n_c * n
    return {"bytes": values * e, "flops": flops}


def tolerance(case):
    # About four times the distance of each path from the same operators in 64 bits on the same inputs:
    # fp32 sums up to 4.5e-7 (one value 5e-6); bf16 towers 2.9e-3 (1.3e-2), attention with its
    # probabilities rounded to bf16 2.9e-3 (2.5e-2), interactions 2.0e-3 (1.0e-2).
    if case["dtype"] == F32:
        return {"rel": 4e-6, "max": 4e-5}
    if case["kind"] in ("dca", "block"):
        return {"rel": 1.2e-2, "max": 1e-1}
    if case["kind"] in ("glm", "fm"):
        return {"rel": 8e-3, "max": 4e-2}
    return {"rel": 1.2e-2, "max": 5e-2}
