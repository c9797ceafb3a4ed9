"""GPU parity: the CUDA kernels, called through the C ABI, against the fp64 CPU oracle.

Error metric for every output tensor: max_i |gpu_i - ref_i| / max_i |ref_i|, which must be
<= 1e-2 for bf16 storage and <= 1e-4 for the fp32 path.  Small cases compare every element;
the full-size configurations compare a stratified sample of candidates (segment ends, the
smallest requests, uniform draws) because the oracle is slow by design.
"""
import ctypes
import time
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest
import torch

from oracle import rocs_ref as ref
from paper_2607_27744_b200 import binding as rocs, workloads as wl
from _util import rel_err, to_dev, to_host_f64, tol_for

pytestmark = pytest.mark.gpu

PATHS = [rocs.PATH_AUTO, rocs.PATH_GENERAL]


@pytest.fixture(autouse=True)
def _reset_path():
    yield
    rocs.set_path(rocs.PATH_AUTO)
    rocs.last_device_status()


def _plan(co):
    return rocs.plan_create(to_dev(co), co)


# ------------------------------------------------------------------ linear ------------------
def _run_linear(cfg, co, bias=False, relu=False, sample=None, path=rocs.PATH_AUTO):
    rocs.set_path(path)
    d = wl.linear_inputs(cfg, co, bias=bias)
    plan = _plan(co)
    W = to_dev(d["W"])
    XR = to_dev(d["XR"]) if cfg.d_req else None
    Y = rocs.ikbo_linear(plan, XR, to_dev(d["XC"]), W[:, :cfg.d_req] if cfg.d_req else None,
                         W[:, cfg.d_req:], bias=to_dev(d["bias"]), relu=relu)
    want = ref.ikbo_linear(co, d["XR"] if cfg.d_req else None, d["XC"], d["W"], bias=d["bias"], relu=relu,
                           sample=sample)
    got = to_host_f64(Y)
    return rel_err(got if sample is None else got[sample], want)


def test_linear_config1_fp32_every_element():
    cfg = wl.CONFIGS[1]
    assert _run_linear(cfg, wl.cand_offsets(cfg), bias=True, relu=True) <= tol_for("f32")


@pytest.mark.parametrize("path", PATHS)
@pytest.mark.parametrize("relu,bias", [(False, False), (True, True)])
def test_linear_bf16_ragged_segments_several_tiles(path, relu, bias):
    # counts straddle the 128-row tiles, include empty and single-candidate requests
    co = wl.offsets_from_counts([1, 0, 127, 129, 300, 0, 2, 513, 64])
    cfg = wl.CONFIGS[2].with_(R=len(co) - 1, d_req=192, d_cand=128, d_out=320)
    assert _run_linear(cfg, co, bias=bias, relu=relu, path=path) <= tol_for("bf16")


@pytest.mark.parametrize("requests,most", [(70, 41), (800, 21)])
@pytest.mark.parametrize("relu,bias", [(False, False), (True, True)])
def test_linear_bf16_narrow_input_many_short_segments(relu, bias, requests, most):
    # 8000 rows with d_cand <= 256 take the weight-stationary kernel, and segments of 0..20 rows put more requests into a run of
    # 256 rows than one launch holds: several in every 32-row slab, so both the shared-memory and the global request rows are
    # exercised; d_out = 328 leaves a ragged last column slice.  1393 rows are one launch of small tiles
    counts = [(i * 7) % most for i in range(requests)]
    co = wl.offsets_from_counts(counts)
    cfg = wl.CONFIGS[5].with_(R=len(counts), d_req=64, d_cand=200, d_out=328)
    assert _run_linear(cfg, co, bias=bias, relu=relu) <= tol_for("bf16")


@pytest.mark.parametrize("path", PATHS)
def test_linear_bf16_odd_widths(path):
    co = wl.offsets_from_counts([5, 77, 1])
    cfg = wl.CONFIGS[2].with_(R=3, d_req=72, d_cand=40, d_out=24)
    assert _run_linear(cfg, co, relu=True, path=path) <= tol_for("bf16")


@pytest.mark.parametrize("path", PATHS)
def test_linear_bf16_no_request_half(path):
    co = wl.offsets_from_counts([200, 56])
    cfg = wl.CONFIGS[2].with_(R=2, d_req=0, d_cand=256, d_out=256)
    assert _run_linear(cfg, co, bias=True, relu=True, path=path) <= tol_for("bf16")


@pytest.mark.parametrize("relu,bias", [(False, True), (True, False)])
def test_plain_linear_bf16_wide_many_rows(relu, bias):
    # M >= 2048 rows, wide K and d_out >= 256 take the CTA-pair K-ring GEMM; M is not a multiple of the
    # 256-row super-tile and d_out = 328 leaves a ragged last column tile
    g = np.random.default_rng(17)
    M, d_in, d_out = 2500, 712, 328
    X = wl.store(g.standard_normal((M, d_in), dtype=np.float32), "bf16")
    W = wl.store(g.standard_normal((d_out, d_in), dtype=np.float32) * d_in ** -0.5, "bf16")
    b = g.standard_normal(d_out).astype(np.float32) if bias else None
    y = rocs.linear(to_dev(X), to_dev(W), bias=to_dev(b), relu=relu)
    want = ref.ikbo_linear(wl.offsets_from_counts([M]), None, X, W, bias=b, relu=relu)
    assert rel_err(to_host_f64(y), want) <= tol_for("bf16")


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("M,d_in,d_out", [(1, 3, 1), (35, 19, 17), (33, 130, 1024), (600, 100, 397), (2600, 35, 517)])
def test_linear_general_kernel_tiles(dtype, M, d_in, d_out):
    # the three tile sizes (16, 32, 64), each with remainders in rows, columns and K; rows padded to 16 bytes
    # with NaN behind the last column, which must not be read into the sum
    rocs.set_path(rocs.PATH_GENERAL)
    g = np.random.default_rng(M)
    X, W = g.standard_normal((M, d_in), dtype=np.float32), g.standard_normal((d_out, d_in), dtype=np.float32)
    b = g.standard_normal(d_out).astype(np.float32)
    X, W = wl.store(X, dtype), wl.store(W * d_in ** -0.5, dtype)
    ld = rocs.padded_ld(d_in, rocs.BF16 if dtype == "bf16" else rocs.F32)

    def padded(a):
        t = torch.full((a.shape[0], ld), float("nan"), dtype=torch.bfloat16 if dtype == "bf16" else torch.float32, device="cuda")
        t[:, :d_in] = to_dev(a)
        return t[:, :d_in]

    ldo = rocs.padded_ld(d_out, rocs.BF16 if dtype == "bf16" else rocs.F32)
    Y = torch.empty((M, ldo), dtype=torch.bfloat16 if dtype == "bf16" else torch.float32, device="cuda")[:, :d_out]
    rocs.linear(padded(X), padded(W), bias=to_dev(b), relu=True, out=Y)
    want = ref.ikbo_linear(wl.offsets_from_counts([M]), None, X, W, bias=b, relu=True)
    assert rel_err(to_host_f64(Y), want) <= tol_for(dtype)


@pytest.mark.parametrize("M,d_out", [(2048, 256), (4866, 1024), (4866, 256), (2305, 520), (9000, 456)])
def test_plain_linear_tile_widths(M, d_out):
    # 128, 192 and 256 columns per tile of the CTA-pair kernel, with and without a partial last tile
    g = np.random.default_rng(M + d_out)
    X = wl.store(g.standard_normal((M, 136), dtype=np.float32), "bf16")
    W = wl.store(g.standard_normal((d_out, 136), dtype=np.float32) * 136 ** -0.5, "bf16")
    b = g.standard_normal(d_out).astype(np.float32)
    y = rocs.linear(to_dev(X), to_dev(W), bias=to_dev(b), relu=True)
    want = ref.ikbo_linear(wl.offsets_from_counts([M]), None, X, W, bias=b, relu=True)
    assert rel_err(to_host_f64(y), want) <= tol_for("bf16")


@pytest.mark.parametrize("N", [1, 7, 9, 127, 129, 500, 511, 16384, 16385])
def test_linear_few_rows_and_both_request_maps(N):
    # X tiles of fewer than 128 rows, both halves in one launch (few requests per tile or run of rows), on small tiles
    # below 512 rows and on CTA pairs
    counts = [0, N // 3, 1, 0, N - N // 3 - 1, 0] if N > 1 else [0, 1]
    co = wl.offsets_from_counts(counts)
    cfg = wl.CONFIGS[2].with_(R=len(counts), d_req=136, d_cand=320 if N < 512 else 72, d_out=192)
    assert _run_linear(cfg, co, bias=True, relu=True) <= tol_for("bf16")


@pytest.mark.parametrize("M", [1, 9, 127, 130, 500])
@pytest.mark.parametrize("d_in,d_out", [(256, 64), (264, 8), (520, 132), (1024, 60), (1048, 256), (2056, 68), (136, 1100)])
def test_plain_linear_small_tiles(M, d_in, d_out):
    # 32, 64 and 128 rows by 32 and 64 columns per tile, ragged last tiles in every dimension
    g = np.random.default_rng(17 * M + d_in)
    X = wl.store(g.standard_normal((M, d_in), dtype=np.float32), "bf16")
    W = wl.store(g.standard_normal((d_out, d_in), dtype=np.float32) * d_in ** -0.5, "bf16")
    b = g.standard_normal(d_out).astype(np.float32)
    ld = rocs.padded_ld(d_out, rocs.BF16)
    y = torch.zeros((M, ld), dtype=torch.bfloat16, device="cuda")
    rocs.linear(to_dev(X), to_dev(W), bias=to_dev(b), relu=True, out=y[:, :d_out])
    want = ref.ikbo_linear(wl.offsets_from_counts([M]), None, X, W, bias=b, relu=True)
    assert rel_err(to_host_f64(y[:, :d_out]), want) <= tol_for("bf16")
    assert torch.all(y[:, d_out:] == 0)


@pytest.mark.parametrize("N", [1, 40, 129, 300])
def test_linear_halves_in_small_tiles(N):
    # a request half longer than the candidate half, in one launch
    counts = [0, N // 3, 1, 0, N - N // 3 - 1, 0] if N > 1 else [0, 1]
    co = wl.offsets_from_counts(counts)
    cfg = wl.CONFIGS[2].with_(R=len(counts), d_req=1032, d_cand=520, d_out=200)
    assert _run_linear(cfg, co, bias=True, relu=True) <= tol_for("bf16")


@pytest.mark.parametrize("N", [2, 33, 127, 500])
@pytest.mark.parametrize("d_req,d_cand", [(136, 72), (136, 320), (1032, 520)])
def test_linear_halves_apart_in_small_tiles(N, d_req, d_cand):
    # a run of 150 requests without candidates inside a tile, more than its rows: the halves are two launches, the candidate
    # half waits for the request half in its epilogue only and searches the request in the offsets
    counts = [0, N // 2, *[0] * 150, N - N // 2, 0]
    co = wl.offsets_from_counts(counts)
    cfg = wl.CONFIGS[2].with_(R=len(counts), d_req=d_req, d_cand=d_cand, d_out=192)
    assert _run_linear(cfg, co, bias=True, relu=True) <= tol_for("bf16")


def _counts_of(law, N, rng):
    if law == "one":
        return [N]
    per = {"each": 1, "few": 6, "many": 300, "gaps": 40}[law]
    counts = []
    while sum(counts) < N:
        counts.append(min(N - sum(counts), int(rng.integers(1, 2 * per)) if per > 1 else 1))
        counts += [0] * int(rng.integers(0, 5)) if law == "gaps" else []
    return [0, 0, *counts, 0] if law == "gaps" else counts


@pytest.mark.parametrize("law", ["one", "each", "few", "many", "gaps"])
@pytest.mark.parametrize("dtype,N,d_req,d_cand,d_out", [
    ("bf16", 33, 200, 8, 72), ("bf16", 500, 520, 256, 512), ("bf16", 600, 8, 304, 256), ("bf16", 1100, 72, 264, 1000),   # tiles of their own
    ("bf16", 1300, 520, 64, 1024), ("bf16", 4866, 200, 256, 1024), ("bf16", 20000, 64, 128, 328), ("bf16", 9500, 768, 8, 64),  # CTA pairs
    ("f32", 1, 3, 5, 9), ("f32", 40, 65, 16, 300), ("f32", 300, 20, 40, 132)])
def test_linear_halves_in_one_launch(dtype, N, d_req, d_cand, d_out, law):
    # the request half in the candidates' launch: one request, as many as rows, so many or so spread out (empty ones
    # in between) that some tiles or runs hold more than fit and the halves are two launches after all
    co = wl.offsets_from_counts(_counts_of(law, N, np.random.default_rng(N)))
    cfg = wl.CONFIGS[5].with_(R=len(co) - 1, dtype=dtype, d_req=d_req, d_cand=d_cand, d_out=d_out)
    ends = np.concatenate([co[:-1], co[1:] - 1, np.arange(0, N, 97), np.arange(0, N, 256)])
    sample = np.unique(np.clip(ends, 0, N - 1))[:1200]
    if dtype == "f32" and (d_req * 4) % 16:
        d = wl.linear_inputs(cfg, co, bias=True)
        def rows(a):  # rows that start on 16-byte boundaries
            t = torch.zeros(a.shape[0], (a.shape[1] + 3) // 4 * 4, device="cuda")
            t[:, :a.shape[1]] = to_dev(a)
            return t[:, :a.shape[1]]
        Y = rocs.ikbo_linear(_plan(co), rows(d["XR"]), rows(d["XC"]), rows(d["W"][:, :d_req]), rows(d["W"][:, d_req:]), bias=to_dev(d["bias"]),
                             out=rows(np.zeros((N, d_out), np.float32)))
        assert rel_err(to_host_f64(Y), ref.ikbo_linear(co, d["XR"], d["XC"], d["W"], bias=d["bias"])) <= tol_for(dtype)
        return
    assert _run_linear(cfg, co, bias=True, relu=law == "few", sample=sample) <= tol_for(dtype)


def test_linear_empty_batch():
    co = np.zeros(3, np.int32)
    cfg = wl.CONFIGS[2].with_(R=2, d_req=64, d_cand=64, d_out=64)
    plan = _plan(co)
    d = wl.linear_inputs(cfg, co)
    W = to_dev(d["W"])
    Y = rocs.ikbo_linear(plan, to_dev(d["XR"]), torch.empty((0, 64), dtype=torch.bfloat16, device="cuda"),
                         W[:, :64], W[:, 64:])
    assert Y.shape == (0, 64)


def test_linear_config2_shapes_reduced_rows():
    # full widths of config 2 (512 | 256 -> 1024), fewer requests so the oracle finishes in seconds
    cfg = wl.CONFIGS[2].with_(R=5, count_const=150)
    assert _run_linear(cfg, wl.cand_offsets(cfg), relu=True) <= tol_for("bf16")


def test_mlp_config2_three_layers_reduced_rows():
    cfg = wl.CONFIGS[2].with_(R=3, count_const=100)
    co = wl.cand_offsets(cfg)
    d = wl.linear_inputs(cfg, co)
    ws = wl.mlp_weights(cfg)
    plan = _plan(co)
    W = to_dev(d["W"])
    h = rocs.ikbo_linear(plan, to_dev(d["XR"]), to_dev(d["XC"]), W[:, :cfg.d_req], W[:, cfg.d_req:], relu=True)
    h = rocs.linear(h, to_dev(ws[0]), relu=True)
    y = rocs.linear(h, to_dev(ws[1]))
    r = ref.ikbo_linear(co, d["XR"], d["XC"], d["W"], relu=True)
    one = wl.offsets_from_counts([r.shape[0]])
    r = ref.ikbo_linear(one, None, r, wl.to_f64(ws[0]), relu=True)
    r = ref.ikbo_linear(one, None, r, wl.to_f64(ws[1]))
    assert rel_err(to_host_f64(y), r) <= tol_for("bf16")


def test_mlp_config2_full_size_sampled():
    # the whole benchmark step (plan, split layer, two plain layers) at full size; the oracle follows
    # the sampled candidates through all three layers in fp64
    cfg = wl.CONFIGS[2]
    co = wl.cand_offsets(cfg)
    d = wl.linear_inputs(cfg, co)
    ws = wl.mlp_weights(cfg)
    sample = wl.stratified_sample(co, n_uniform=128, n_small_requests=0, cfg_id=2)
    plan = _plan(co)
    W = to_dev(d["W"])
    h = rocs.ikbo_linear(plan, to_dev(d["XR"]), to_dev(d["XC"]), W[:, :cfg.d_req], W[:, cfg.d_req:], relu=True)
    h = rocs.linear(h, to_dev(ws[0]), relu=True)
    y = rocs.linear(h, to_dev(ws[1]))
    r = ref.ikbo_linear(co, d["XR"], d["XC"], d["W"], relu=True, sample=sample)
    one = wl.offsets_from_counts([r.shape[0]])
    r = ref.ikbo_linear(one, None, r, wl.to_f64(ws[0]), relu=True)
    r = ref.ikbo_linear(one, None, r, wl.to_f64(ws[1]))
    assert rel_err(to_host_f64(y)[sample], r) <= tol_for("bf16")


def test_isolation_config2_full_size_is_bit_exact():
    # Eq. 1 at the size and launch configuration the benchmark times: one candidate changes, every
    # other output row of the split layer keeps its bits
    cfg = wl.CONFIGS[2]
    co = wl.cand_offsets(cfg)
    d = wl.linear_inputs(cfg, co)
    plan = _plan(co)
    W, XR, XC = to_dev(d["W"]), to_dev(d["XR"]), to_dev(d["XC"])
    base = rocs.ikbo_linear(plan, XR, XC, W[:, :cfg.d_req], W[:, cfg.d_req:], relu=True)
    j = 77_777
    XC2 = XC.clone()
    XC2[j] += 1.0
    pert = rocs.ikbo_linear(plan, XR, XC2, W[:, :cfg.d_req], W[:, cfg.d_req:], relu=True)
    same = (base.view(torch.int16) == pert.view(torch.int16)).all(dim=1)
    assert not bool(same[j])
    same[j] = True
    assert bool(same.all())


def test_linear_config2_full_size_sampled():
    cfg = wl.CONFIGS[2]
    co = wl.cand_offsets(cfg)
    sample = wl.stratified_sample(co, n_uniform=256, n_small_requests=0, cfg_id=2)
    assert _run_linear(cfg, co, relu=True, sample=sample) <= tol_for("bf16")


def test_linear_config5_full_size_sampled():
    cfg = wl.CONFIGS[5]
    co = wl.cand_offsets(cfg)
    sample = wl.stratified_sample(co, n_uniform=256, n_small_requests=8, cfg_id=5)
    assert _run_linear(cfg, co, sample=sample) <= tol_for("bf16")


# ------------------------------------------------------------------ attention ---------------
def _run_dca(cfg, co, so, sample=None, path=rocs.PATH_AUTO, scale=0.0):
    rocs.set_path(path)
    d = wl.dca_inputs(cfg, co, so)
    plan = _plan(co)
    O = rocs.dca_attention(plan, to_dev(d["Q"]), to_dev(d["K"]), to_dev(d["V"]), to_dev(so), scale=scale)
    want = ref.dca_attention(co, so, d["Q"], d["K"], d["V"], scale=scale if scale > 0 else None, sample=sample)
    got = to_host_f64(O)
    return rel_err(got if sample is None else got[sample], want)


def test_dca_config1_fp32_every_element():
    cfg = wl.CONFIGS[1]
    assert _run_dca(cfg, wl.cand_offsets(cfg), wl.seq_offsets(cfg)) <= tol_for("f32")


@pytest.mark.parametrize("path", PATHS)
def test_dca_bf16_ragged(path):
    # segments around the 128-row tile, empty request, empty sequence, lengths around the key tile
    co = wl.offsets_from_counts([1, 130, 0, 128, 17, 255])
    so = wl.offsets_from_counts([5, 128, 64, 129, 0, 300])
    cfg = wl.CONFIGS[3].with_(R=6, H=2, dh=64)
    assert _run_dca(cfg, co, so, path=path) <= tol_for("bf16")


@pytest.mark.parametrize("path", PATHS)
def test_dca_bf16_several_query_tokens_and_scale(path):
    co = wl.offsets_from_counts([3, 50, 9])
    so = wl.offsets_from_counts([70, 33, 257])
    cfg = wl.CONFIGS[3].with_(R=3, H=3, dh=64, n_q=5)
    assert _run_dca(cfg, co, so, path=path, scale=0.2) <= tol_for("bf16")


def test_dca_bf16_32_query_tokens_per_candidate():
    # the paper's typical candidate-side query length (Section 4.3): four candidates fill a 128-row tile
    co = wl.offsets_from_counts([9, 1, 30])
    so = wl.offsets_from_counts([200, 64, 130])
    cfg = wl.CONFIGS[3].with_(R=3, H=2, dh=64, n_q=32)
    assert _run_dca(cfg, co, so) <= tol_for("bf16")


def test_dca_request_side_query_group():
    # A^R of Eq. 13 (first line) through the same kernel: one query group per request, i.e. a plan
    # whose "candidates" are the requests themselves
    R = 5
    co = np.arange(R + 1, dtype=np.int32)
    so = wl.offsets_from_counts([300, 17, 0, 128, 65])
    cfg = wl.CONFIGS[3].with_(R=R, H=4, dh=64, n_q=16)
    assert _run_dca(cfg, co, so) <= tol_for("bf16")


@pytest.mark.parametrize("dh", [32, 128])
def test_dca_bf16_other_head_dims(dh):
    co = wl.offsets_from_counts([40, 2])
    so = wl.offsets_from_counts([100, 31])
    cfg = wl.CONFIGS[3].with_(R=2, H=2, dh=dh)
    assert _run_dca(cfg, co, so) <= tol_for("bf16")


@pytest.mark.parametrize("dh", [32, 128])
def test_dca_bf16_head_dim_32_and_128_ragged_on_tensor_cores(dh):
    # dh = 128 runs on the tensor-core kernel with 64-key blocks, dh = 32 with 64-byte operand rows:
    # segments around the 128-row tile, empty request / sequence, lengths around the key block, several
    # query tokens
    co = wl.offsets_from_counts([1, 130, 0, 128, 17, 255])
    so = wl.offsets_from_counts([5, 128, 64, 129, 0, 300])
    cfg = wl.CONFIGS[3].with_(R=6, H=2, dh=dh)
    assert _run_dca(cfg, co, so) <= tol_for("bf16")
    cfg = wl.CONFIGS[3].with_(R=3, H=3, dh=dh, n_q=5)
    assert _run_dca(cfg, wl.offsets_from_counts([3, 50, 9]), wl.offsets_from_counts([70, 33, 257]), scale=0.1) <= tol_for("bf16")


@pytest.mark.parametrize("dh", [32, 64, 128])
@pytest.mark.parametrize("R,n,H,L", [(1, 7, 1, 2048), (2, 300, 2, 1500), (3, 129, 4, 1030), (5, 200, 8, 700), (9, 100, 16, 400),
                                     (300, 0, 1, 600), (1, 5, 2, 4000)])
def test_dca_bf16_items_split_along_their_keys(dh, R, n, H, L):
    # clusters of 8, 4, 2 and 1 CTAs, sequences shorter than the batch's average (sides without keys), a request
    # without keys and one without candidates, more requests than a warp has lanes, item list and item search;
    # scores that outgrow the reference of one part only, of all rows but one
    g = np.random.default_rng(R * 7 + n)
    counts = [n if n else int(r % 97 == 5) for r in range(R)]
    lens = [L if r == 0 else int(g.integers(0, 2 * L)) for r in range(R)]
    if R > 2:
        counts[1], lens[2] = 0, 0
    if R > 3:
        lens[3] = 17
    co, so = wl.offsets_from_counts(counts), wl.offsets_from_counts(lens)
    cfg = wl.CONFIGS[3].with_(R=R, H=H, dh=dh)
    assert _run_dca(cfg, co, so) <= tol_for("bf16")
    d = wl.dca_inputs(cfg, co, so)
    if lens[0] > 300 and counts[0] > 4:
        K = wl.bf16_bits_to_f32(d["K"]).copy()
        K[290] = wl.bf16_bits_to_f32(d["Q"])[3, 0] * 60.0
        d["K"] = wl.f32_to_bf16_bits(K)
        want = ref.dca_attention(co, so, d["Q"], d["K"], d["V"])
        O = rocs.dca_attention(_plan(co), to_dev(d["Q"]), to_dev(d["K"]), to_dev(d["V"]), to_dev(so))
        assert rel_err(to_host_f64(O), want) <= tol_for("bf16")


@pytest.mark.parametrize("dh", [32, 64, 128])
def test_dca_bf16_short_last_blocks_between_empty_requests(dh):
    # products of the last key block end at a multiple of 16 keys, the rows of V between are zeroed behind the next
    # item's loads: every remainder class, items with no keys and with no ragged end in between, one item per side
    # and long streams; V rows behind each sequence hold NaN, in a request that has no candidates
    lens = [1, 0, 15, 16, 17, 0, 0, 31, 33, 48, 63, 64, 65, 79, 80, 81, 0, 95, 97, 112, 127, 128, 129, 143, 144, 145, 200, 257]
    co = wl.offsets_from_counts([c for _ in lens for c in (3, 0)])
    so = wl.offsets_from_counts([x for n in lens for x in (n, 3)])
    for H in (1, 16):
        cfg = wl.CONFIGS[3].with_(R=len(co) - 1, H=H, dh=dh)
        d = wl.dca_inputs(cfg, co, so)
        V = wl.bf16_bits_to_f32(d["V"]).copy()
        want = ref.dca_attention(co, so, d["Q"], d["K"], d["V"])
        for r in range(1, len(so) - 1, 2):
            V[so[r]:so[r + 1]] = np.nan
        O = rocs.dca_attention(_plan(co), to_dev(d["Q"]), to_dev(d["K"]), to_dev(wl.f32_to_bf16_bits(V)), to_dev(so))
        assert rel_err(to_host_f64(O), want) <= tol_for("bf16")


@pytest.mark.parametrize("dh", [32, 64, 128])
@pytest.mark.parametrize("heads", [1, 4, 64])
def test_dca_bf16_streams_that_end_with_short_ragged_items(dh, heads):
    # the last item of a side's stream is loaded whole while the one in front of it is still at work; both end
    # inside a group of 16 keys.  Items taken by position (few or very many) and claimed; repeated, since what goes
    # wrong is a hand-over that comes too early
    R = 200
    co = wl.offsets_from_counts([3] * R)
    so = wl.offsets_from_counts([150 + (r * 37) % 90 if r < R // 2 else 1 + (r * 7) % 60 for r in range(R)])
    cfg = wl.CONFIGS[3].with_(R=R, H=heads, dh=dh)
    d = wl.dca_inputs(cfg, co, so)
    Q, K, V, sod, plan = to_dev(d["Q"]), to_dev(d["K"]), to_dev(d["V"]), to_dev(so), _plan(co)
    want = ref.dca_attention(co, so, d["Q"], d["K"], d["V"])
    for _ in range(300):
        O = rocs.dca_attention(plan, Q, K, V, sod)
    assert rocs.last_device_status() == 0
    assert rel_err(to_host_f64(O), want) <= tol_for("bf16")


@pytest.mark.parametrize("dh", [32, 128])
def test_dca_bf16_head_dim_32_and_128_many_tiles_sampled(dh):
    # enough tiles that every SM runs several items on both of its streams (L = 700: 11 or 6 key blocks)
    cfg = wl.CONFIGS[3].with_(R=48, H=4, dh=dh, L_const=700)
    co, so = wl.cand_offsets(cfg), wl.seq_offsets(cfg)
    sample = wl.stratified_sample(co, n_uniform=128, n_small_requests=2, cfg_id=3)
    assert _run_dca(cfg, co, so, sample=sample) <= tol_for("bf16")


@pytest.mark.parametrize("dh", [32, 64, 128])
def test_dca_bf16_scores_that_outgrow_the_first_key_block(dh):
    # The tensor-core kernel fixes a row's softmax reference from its first key block.  Keys far
    # down the sequence that are large multiples of a query row push that row's (and, through
    # chance alignment, other rows') scores hundreds of nats above the reference, beyond what
    # fp32 exponentials can hold: such rows must come out of the kernel's plain-fp32 recomputation,
    # and every other row must be untouched by it.
    co = wl.offsets_from_counts([200, 100])
    so = wl.offsets_from_counts([600, 300])
    cfg = wl.CONFIGS[5].with_(R=2, dh=dh)
    d = wl.dca_inputs(cfg, co, so)
    Q, K = wl.bf16_bits_to_f32(d["Q"]), wl.bf16_bits_to_f32(d["K"])
    K[300] = Q[5, 0] * 60.0      # request 0, third key block: +60 |q|^2 for query row 5
    K[450] = Q[140, 0] * 3.0
    K[258] = Q[7, 0] * 60.0
    K[130] = Q[150, 0] * -80.0   # second key block: huge negative for row 150, +-hundreds for the rest
    K[700] = Q[250, 0] * 40.0    # request 1, second key block
    d["K"] = wl.f32_to_bf16_bits(K)
    plan = _plan(co)
    O = rocs.dca_attention(plan, to_dev(d["Q"]), to_dev(d["K"]), to_dev(d["V"]), to_dev(so))
    want = ref.dca_attention(co, so, d["Q"], d["K"], d["V"])
    assert rel_err(to_host_f64(O), want) <= tol_for("bf16")
    assert rocs.last_device_status() == 0


@pytest.mark.parametrize("dtype,dh,n_q", [("f32", 4, 1), ("f32", 36, 3), ("f32", 64, 70), ("f32", 128, 1), ("f32", 200, 1),
                                          ("bf16", 96, 1), ("bf16", 256, 2)])
def test_dca_general_kernel_edges(dtype, dh, n_q):
    # tiles of 32 query rows and 64 keys: one row / key, one less, exact, one more; empty request and sequence;
    # head widths between the compiled ones; more query tokens than a tile has rows
    co = wl.offsets_from_counts([1, 31, 32, 0, 65, 2] if n_q < 64 else [1, 0, 2, 1, 1, 3])
    so = wl.offsets_from_counts([63, 64, 1, 40, 129, 0])
    cfg = wl.CONFIGS[3].with_(R=6, H=3, dh=dh, n_q=n_q, dtype=dtype)
    assert _run_dca(cfg, co, so) <= tol_for(dtype)


@pytest.mark.parametrize("dh", [20, 64])
@pytest.mark.parametrize("L", [64, 65, 128, 129, 300])
def test_dca_general_kernel_groups_of_keys(L, dh):
    # one group of threads or two per tile, the second without keys, with a part of a block, with another number of
    # blocks than the first; between requests with few keys or none; a first block whose scores are all -inf
    lengths = np.array([L, 3, 0, 2 * L - 70 if L > 64 else 63, L], np.int32)
    so = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    co = wl.offsets_from_counts([5, 1, 2, 33, 4])
    cfg = wl.CONFIGS[1].with_(R=5, H=2, dh=dh)
    d = wl.dca_inputs(cfg, co, so)
    d["Q"][-4:, ..., 0] = 1.0
    d["K"][so[4]:so[4] + 64, :, 0] = -np.inf
    O = rocs.dca_attention(_plan(co), to_dev(d["Q"]), to_dev(d["K"]), to_dev(d["V"]), to_dev(so))
    want = ref.dca_attention(co, so, d["Q"], d["K"], d["V"])
    if L == 64:  # of these rows every score is -inf
        assert bool(torch.isnan(O[-4:]).all())
        O, want = O[:-4], want[:-4]
    assert rel_err(to_host_f64(O), want) <= tol_for("f32")


@pytest.mark.parametrize("R", [12, 33, 64, 65])
def test_dca_bf16_items_by_length(R):
    # up to 64 requests with long sequences: items in the order of their number of keys, from none to several times the
    # average, requests without candidates in between; one more request and the order is that of the requests
    g = np.random.default_rng(R)
    lengths = g.choice([0, 1, 130, 640, 700, 1400, 2500], R)
    lengths[0] = 3000
    counts = g.integers(0, 36000 // R, R) * (g.random(R) < 0.8)
    counts[-1] = 500
    co, so = wl.offsets_from_counts(counts.tolist()), np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    cfg = wl.CONFIGS[3].with_(R=R, H=4, dh=128)
    N = int(co[-1])
    sample = np.unique(np.concatenate([np.clip(np.stack([co[:-1], co[1:] - 1]).ravel(), 0, N - 1), g.integers(0, N, 150)]))
    assert _run_dca(cfg, co, so, sample=sample) <= tol_for("bf16")


def test_dca_bf16_64_query_tokens_per_candidate():
    # two candidates fill a 128-row tile (Section 4.3.2 names query tiles of 32 and 64 tokens)
    co = wl.offsets_from_counts([5, 1, 12, 2])
    so = wl.offsets_from_counts([200, 64, 130, 513])
    cfg = wl.CONFIGS[3].with_(R=4, H=2, dh=64, n_q=64)
    assert _run_dca(cfg, co, so) <= tol_for("bf16")


def test_dca_config3_shapes_reduced_requests():
    cfg = wl.CONFIGS[3].with_(R=2)
    co = wl.offsets_from_counts([140, 9])
    assert _run_dca(cfg, co, wl.seq_offsets(cfg)) <= tol_for("bf16")


def test_dca_stack_config3_two_layers_reduced():
    # h_0 = x^C; Q_l = W_Q,l h_{l-1}; A_l = DCA(Q_l, K_l, V_l); h_l = [h_{l-1}, A_l]
    cfg = wl.CONFIGS[3].with_(R=2, L_const=200)
    co = wl.offsets_from_counts([70, 3])
    so = wl.seq_offsets(cfg)
    d = wl.dca_stack_inputs(cfg, co, so)
    plan = _plan(co)
    N = int(co[-1])
    h = to_dev(d["XC"])
    hr = wl.to_f64(d["XC"])
    one = wl.offsets_from_counts([N])
    for lay in d["layers"]:
        q = rocs.linear(h, to_dev(lay["WQ"]))
        a = rocs.dca_attention(plan, q.view(N, 1, cfg.H, cfg.dh), to_dev(lay["K"]), to_dev(lay["V"]), to_dev(so))
        h = torch.cat([h, a.view(N, -1)], dim=1).contiguous()
        qr = ref.ikbo_linear(one, None, hr, wl.to_f64(lay["WQ"]))
        ar = ref.dca_attention(co, so, qr.reshape(N, 1, cfg.H, cfg.dh), wl.to_f64(lay["K"]), wl.to_f64(lay["V"]))
        hr = np.concatenate([hr, ar.reshape(N, -1)], axis=1)
    assert rel_err(to_host_f64(h), hr) <= tol_for("bf16")


def test_dca_stack_config3_full_size_sampled():
    # two stacked DCA layers at full size: Q_l = W_Q,l h_{l-1}, A_l = DCA(Q_l, K_l, V_l), h_l = [h_{l-1}, A_l];
    # the oracle follows a sample of candidates through both layers
    cfg = wl.CONFIGS[3]
    co, so = wl.cand_offsets(cfg), wl.seq_offsets(cfg)
    d = wl.dca_stack_inputs(cfg, co, so)
    plan = _plan(co)
    N = int(co[-1])
    sample = wl.stratified_sample(co, n_uniform=24, n_small_requests=0, cfg_id=3)[::4]
    h = to_dev(d["XC"])
    hr = wl.to_f64(d["XC"])[sample]
    one = wl.offsets_from_counts([sample.size])
    for lay in d["layers"]:
        q = rocs.linear(h, to_dev(lay["WQ"]))
        a = rocs.dca_attention(plan, q.view(N, 1, cfg.H, cfg.dh), to_dev(lay["K"]), to_dev(lay["V"]), to_dev(so))
        h = torch.cat([h, a.view(N, -1)], dim=1).contiguous()
        qr = ref.ikbo_linear(one, None, hr, wl.to_f64(lay["WQ"]))
        # the oracle attends the sampled rows against their own requests: scatter them into a full-size Q
        Qf = np.zeros((N, 1, cfg.H, cfg.dh))
        Qf[sample] = qr.reshape(-1, 1, cfg.H, cfg.dh)
        ar = ref.dca_attention(co, so, Qf, wl.to_f64(lay["K"]), wl.to_f64(lay["V"]), sample=sample)
        hr = np.concatenate([hr, ar.reshape(sample.size, -1)], axis=1)
    assert rel_err(to_host_f64(h)[sample], hr) <= tol_for("bf16")


def test_dca_config3_full_size_sampled():
    cfg = wl.CONFIGS[3]
    co, so = wl.cand_offsets(cfg), wl.seq_offsets(cfg)
    sample = wl.stratified_sample(co, n_uniform=64, n_small_requests=1, cfg_id=3)
    assert _run_dca(cfg, co, so, sample=sample) <= tol_for("bf16")


def test_dca_config5_full_size_sampled():
    cfg = wl.CONFIGS[5]
    co, so = wl.cand_offsets(cfg), wl.seq_offsets(cfg)
    sample = wl.stratified_sample(co, n_uniform=128, n_small_requests=4, cfg_id=5)
    assert _run_dca(cfg, co, so, sample=sample) <= tol_for("bf16")


@pytest.mark.parametrize("L", [200, 1500])   # one part per item; split over sides and CTAs
@pytest.mark.parametrize("dh", [32, 64, 128])
@pytest.mark.parametrize("where", ["head", "tail", "most", "all"])
def test_dca_bf16_scores_of_minus_infinity(L, dh, where):
    # a key whose score is -inf has weight 0, also where all keys of a part score so; a row of nothing else is NaN
    co, so = wl.offsets_from_counts([40, 0, 3]), wl.offsets_from_counts([L, 5, L - 37])
    cfg = wl.CONFIGS[3].with_(R=3, H=2, dh=dh)
    d = wl.dca_inputs(cfg, co, so)
    Q, K, V = to_dev(d["Q"]), to_dev(d["K"]), to_dev(d["V"])
    Q[..., 0] = Q[..., 0].abs() + 0.5
    for r in (0, 2):
        n = int(so[r + 1] - so[r])
        keys = {"head": slice(0, n // 2), "tail": slice(n // 3, n), "most": slice(0, n - 1), "all": slice(0, n)}[where]
        K[int(so[r]):int(so[r + 1])][keys, :, 0] = float("-inf")
    got = rocs.dca_attention(_plan(co), Q, K, V, to_dev(so)).double()
    if where == "all":
        assert bool(torch.isnan(got).all())
        return
    want = torch.empty_like(got)
    for r in (0, 2):
        c, k = slice(int(co[r]), int(co[r + 1])), slice(int(so[r]), int(so[r + 1]))
        p = torch.softmax(torch.einsum("nqhd,khd->nqhk", Q[c].double(), K[k].double()) * dh ** -0.5, -1)
        want[c] = torch.einsum("nqhk,khd->nqhd", p, V[k].double())
    assert rel_err(got.cpu().numpy(), want.cpu().numpy()) <= tol_for("bf16")


@pytest.mark.parametrize("dh", [32, 64, 128])
@pytest.mark.parametrize("log2_weight", [126, 123])
def test_dca_bf16_split_items_whose_parts_add_up_past_fp32(dh, log2_weight):
    # The last key of every 128 weighs 2^126 against the reference 1 of its part: three of them are within fp32 in each of
    # 4 parts (8 at width 128), a dozen are not.  The rows are the mean of these keys' values.
    co, so = wl.offsets_from_counts([40, 3]), wl.offsets_from_counts([1536, 1536])
    Q = torch.zeros((43, 1, 2, dh), dtype=torch.bfloat16, device="cuda")
    K = torch.zeros((3072, 2, dh), dtype=torch.bfloat16, device="cuda")
    V = (torch.randn((3072, 2, dh), generator=torch.Generator().manual_seed(3)) * 0.05).to(torch.bfloat16).cuda()
    Q[..., 0] = 1.0
    K[127::128, :, 0] = log2_weight
    got = rocs.dca_attention(_plan(co), Q, K, V, to_dev(so), scale=float(np.log(2.0)))
    want = torch.stack([V[127:1536:128].double().mean(0)] * 40 + [V[1536 + 127::128].double().mean(0)] * 3)[:, None]
    assert rel_err(to_host_f64(got), want.cpu().numpy()) <= tol_for("bf16")


# ------------------------------------------------------------------ interaction -------------
def _run_glm(cfg, co, sample=None, path=rocs.PATH_AUTO):
    rocs.set_path(path)
    d = wl.glm_inputs(cfg, co)
    plan = _plan(co)
    outs = rocs.glm_interaction(plan, to_dev(d["XR"]), to_dev(d["XC"]), to_dev(d["W"]), cfg.n_ro, cfg.n_co)
    G, O = ref.glm_interaction(co, d["XR"], d["XC"], d["W"], cfg.n_ro, cfg.n_co, sample=sample)
    m = np.repeat(np.arange(cfg.R), np.diff(co))
    sel = (lambda a: a) if sample is None else (lambda a: a[sample])
    errs = []
    if G.shape[0]:
        errs.append(rel_err(sel(to_host_f64(outs["YC"])), G[:, cfg.n_r:]))
        errs.append(rel_err(sel(to_host_f64(outs["YR"])[m]), G[:, :cfg.n_r]))
        if O is not None:
            errs.append(rel_err(sel(to_host_f64(outs["OC"])), O[:, cfg.n_ro:]))
            errs.append(rel_err(sel(to_host_f64(outs["OR"])[m]), O[:, :cfg.n_ro]))
    return max(errs) if errs else 0.0


def test_glm_config1_fp32_every_element():
    cfg = wl.CONFIGS[1].with_(n_ro=3, n_co=2)
    assert _run_glm(cfg, wl.cand_offsets(cfg)) <= tol_for("f32")


@pytest.mark.parametrize("path", PATHS)
@pytest.mark.parametrize("which", [4, 5])
def test_glm_bf16_ragged(path, which):
    co = wl.offsets_from_counts([1, 0, 9, 8, 33, 7, 130])
    cfg = wl.CONFIGS[which].with_(R=len(co) - 1)
    if which == 5:
        cfg = cfg.with_(n_ro=0, n_co=0)
    assert _run_glm(cfg, co, path=path) <= tol_for("bf16")


@pytest.mark.parametrize("path", PATHS)
@pytest.mark.parametrize("per", [20, 200])
def test_glm_bf16_other_split(path, per):
    # 203 candidates are more products than the general kernels take of themselves
    co = wl.offsets_from_counts([per, 3])
    cfg = wl.CONFIGS[4].with_(R=2, n_r=16, n_c=16, d_emb=64, n_ro=4, n_co=12)
    assert _run_glm(cfg, co, path=path) <= tol_for("bf16")


@pytest.mark.parametrize("dtype,n_r,n_c,d,n_co", [("f32", 4, 2, 16, 0), ("f32", 1, 1, 4, 1), ("f32", 30, 7, 20, 5), ("f32", 24, 8, 128, 4),
                                                   ("f32", 5, 70, 12, 3), ("f32", 8, 220, 4, 64), ("bf16", 20, 12, 72, 6), ("bf16", 3, 5, 8, 9)])
def test_glm_general_kernel_tiles(dtype, n_r, n_c, d, n_co):
    # tiles of about 64 rows: several candidates, one candidate wider than a tile, embedding counts that leave
    # remainders in every 4 x 4 group, a compression block too large for shared memory
    co = wl.offsets_from_counts([1, 0, 9, 33, 2] if n_c < 100 else [1, 0, 3])
    cfg = wl.CONFIGS[4].with_(R=len(co) - 1, dtype=dtype, n_r=n_r, n_c=n_c, d_emb=d, n_ro=min(2, n_co), n_co=n_co)
    assert _run_glm(cfg, co) <= tol_for(dtype)


@pytest.mark.parametrize("R", [1, 3, 128, 129])
@pytest.mark.parametrize("per", [1, 31, 600])
@pytest.mark.parametrize("dtype,n_r,n_c,d,n_co", [("f32", 32, 2, 128, 8), ("f32", 24, 8, 36, 5), ("bf16", 30, 2, 64, 4), ("f32", 9, 3, 8, 0)])
def test_glm_general_kernel_batch_sizes(dtype, n_r, n_c, d, n_co, per, R):
    # tiles of one candidate up to 64 rows, lanes that share a product or not, the request side in the same launch or
    # (more requests than the blocks look through, or more tiles) in one of its own
    co = wl.offsets_from_counts([per if R < 100 else 1 + r % 5 for r in range(R)])
    cfg = wl.CONFIGS[4].with_(R=R, dtype=dtype, n_r=n_r, n_c=n_c, d_emb=d, n_ro=min(3, n_co), n_co=n_co)
    assert _run_glm(cfg, co) <= tol_for(dtype)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_glm_small_batch_behind_the_kernel_that_writes_its_rows(dtype):
    # the interaction's only launch may start while the kernel in front of it still writes X^R and X^C
    co = wl.offsets_from_counts([7, 1, 12])
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    plan, d, n_r, n_c = _plan(co), 64, 20, 4
    gen = torch.Generator(device="cuda").manual_seed(3)
    W = torch.randn(8, n_r + n_c, device="cuda", generator=gen).to(dt)
    ER, EC = torch.empty(3, n_r, d, dtype=dt, device="cuda"), torch.empty(20, n_c, d, dtype=dt, device="cuda")
    ws = torch.empty(rocs.glm_interaction_workspace(plan, n_r, n_c, 4), dtype=torch.uint8, device="cuda")
    raw = [(torch.randn(3 * n_r, d, device="cuda", generator=gen).to(dt), torch.randn(20 * n_c, d, device="cuda", generator=gen).to(dt)) for _ in range(20)]
    got = []
    for r, c in raw:
        rocs.group_norm(r, out=ER.view(-1, d))
        rocs.group_norm(c, out=EC.view(-1, d))
        got.append({k: v.clone() for k, v in rocs.glm_interaction(plan, ER, EC, W, 4, 4, want_raw=True, workspace=ws).items()})
    for (r, c), out in zip(raw, got):
        rocs.group_norm(r, out=ER.view(-1, d))
        rocs.group_norm(c, out=EC.view(-1, d))
        torch.cuda.synchronize()
        want = rocs.glm_interaction(plan, ER, EC, W, 4, 4, want_raw=True, workspace=ws)
        for k in want:
            assert torch.equal(out[k], want[k]), k


@pytest.mark.parametrize("n_r,n_c,d,n_co,raw", [(32, 16, 128, 8, False), (20, 12, 64, 4, True), (4, 4, 192, 16, True), (44, 8, 256, 3, False),
                                                  (20, 8, 128, 0, True), (16, 4, 64, 8, False), (100, 16, 64, 16, True),
                                                  (128, 12, 256, 1, False), (44, 16, 128, 0, True), (24, 12, 128, 8, False)])
@pytest.mark.parametrize("many", [False, True])
def test_glm_fragments(n_r, n_c, d, n_co, raw, many):
    # 4 to 16 embeddings per candidate (one to four candidates per 16-row fragment, unused rows in some), request
    # columns that end inside a group of 16 and take several passes, fewer fragments than warps; a candidate
    # and a request full of NaN must show in their own rows only
    counts = [1, 0, 9, 8, 33, 7, 0, 133] * (30 if many else 1)
    counts += [3000] if many and n_c < 8 else [0] * 125  # (few products of up to 128 requests are the general kernels')
    co = wl.offsets_from_counts(counts)
    cfg = wl.CONFIGS[4].with_(R=len(co) - 1, n_r=n_r, n_c=n_c, d_emb=d, n_ro=min(2, n_co), n_co=n_co)
    g = wl.glm_inputs(cfg, co)
    plan, W = _plan(co), to_dev(g["W"]) if n_co else None
    N, m = int(co[-1]), np.repeat(np.arange(cfg.R), np.diff(co))

    def run(XR, XC):
        o = rocs.glm_interaction(plan, to_dev(XR), to_dev(XC), W, cfg.n_ro, cfg.n_co, want_raw=raw)
        return {k: o[k] for k in ("YC", "OC") if k in o}

    base = run(g["XR"], g["XC"])
    sample = np.unique(np.concatenate([np.arange(min(N, 70)), np.random.default_rng(1).integers(0, N, 60), [N - 1]]))
    G, O = ref.glm_interaction(co, g["XR"], g["XC"], g["W"] if n_co else None, cfg.n_ro, cfg.n_co, sample=sample)
    if raw:
        assert rel_err(to_host_f64(base["YC"])[sample], G[:, n_r:]) <= tol_for("bf16")
    if n_co:
        assert rel_err(to_host_f64(base["OC"])[sample], O[:, cfg.n_ro:]) <= tol_for("bf16")
    XC, XR = g["XC"].copy(), g["XR"].copy()
    XC[12], XR[4] = 0x7fc0, 0x7fc0
    pert = run(XR, XC)
    keep = (m != 4) & (np.arange(N) != 12)
    for k in base:
        assert np.array_equal(_bits(base[k])[keep], _bits(pert[k])[keep])
        assert bool(torch.isnan(pert[k][12].float()).any())


@pytest.mark.parametrize("n_r,n_c,d,n_co,raw", [(20, 12, 128, 4, False), (16, 4, 64, 8, True), (44, 8, 256, 3, False), (100, 16, 64, 16, True)])
def test_glm_fragments_are_as_exact_as_fp32_arithmetic(n_r, n_c, d, n_co, raw):
    # Both kernels compress the fp32 products and round the result to bf16 once.  Sums of fp32 in another order differ by
    # some 2^-20, against the 2^-9 of that rounding: the errors against fp64 are the same up to which way close values are
    # rounded (well below 1 % of the norm over these thousands of values; products rounded first would add about 20 %).
    co = wl.offsets_from_counts([1, 0, 9, 8, 33, 7, 0, 133] + [0] * 125)  # (few products of up to 128 requests are one kernel on both paths)
    cfg = wl.CONFIGS[4].with_(R=len(co) - 1, n_r=n_r, n_c=n_c, d_emb=d, n_ro=2, n_co=n_co)
    g = wl.glm_inputs(cfg, co)
    want = ref.glm_interaction(co, g["XR"], g["XC"], g["W"], cfg.n_ro, n_co)[1][:, cfg.n_ro:]
    plan = _plan(co)

    def run(XC, W):
        return to_host_f64(rocs.glm_interaction(plan, to_dev(g["XR"]), to_dev(XC), to_dev(W), 2, n_co, want_raw=raw)["OC"])

    XC, W = g["XC"].copy(), g["W"].copy()
    XC[60, 1, 5] = 0x7f80                          # infinities show in the same values either way
    W[cfg.n_ro + n_co - 1, n_r + n_c - 1] = 0xff80
    err, kinds, values = [], [], []
    for path in PATHS:
        rocs.set_path(path)
        got = run(g["XC"], g["W"])
        values.append(got)
        err.append(np.linalg.norm(got - want) / np.linalg.norm(want))
        kinds.append([np.where(np.isnan(o), 2, np.where(np.isinf(o), np.sign(o), 0)) for o in (run(XC, g["W"]), run(g["XC"], W))])
    assert not np.array_equal(*values), "the same kernel on both paths"
    assert err[0] <= 1.01 * err[1]
    for auto, general in zip(*kinds):
        assert np.array_equal(auto, general) and np.any(auto[60] != 0)


@pytest.mark.parametrize("R", [1, 127, 128, 129, 255, 257, 12000, 12001])
def test_work_lists_of_many_requests(R):
    # the lists are scanned by 256 threads per block up to 12000 requests and on the host beyond: counts of
    # 0..3 candidates put empty requests at both ends of every thread's share
    co = wl.offsets_from_counts([(i * 5 + 3) % 4 for i in range(R)])
    # (48 embeddings of up to 128 requests: with 8 so few products are the general kernels')
    assert _run_glm(wl.CONFIGS[5].with_(R=R, n_r=48 if R <= 128 else 8, d_emb=64, n_ro=0, n_co=0), co) <= tol_for("bf16")
    so = wl.offsets_from_counts([(i * 3) % 5 for i in range(R)])
    assert _run_dca(wl.CONFIGS[3].with_(R=R, H=2, dh=8), co, so) <= tol_for("bf16")
    assert _run_dca(wl.CONFIGS[3].with_(R=R, H=2, dh=32), co, so) <= tol_for("bf16")


@pytest.mark.parametrize("R", [1, 31, 33, 200, 512])
@pytest.mark.parametrize("n_c", [8, 12])
def test_glm_tiles_walked_in_the_offsets(R, n_c):
    # runs of tiles that begin and end inside requests, behind partial last tiles and runs of empty requests
    g = np.random.default_rng(R)
    co = wl.offsets_from_counts([int(c) for c in g.choice([0, 0, 1, 7, 16, 17, 40], R - 1)] + [23 if R > 128 else 623])  # (more products than the general kernels take)
    assert _run_glm(wl.CONFIGS[5].with_(R=R, n_r=8, n_c=n_c, d_emb=64, n_ro=2, n_co=4), co) <= tol_for("bf16")


@pytest.mark.parametrize("R,most", [(150, 16), (60, 400)])
@pytest.mark.parametrize("n_r,n_c,d,n_co", [(32, 16, 128, 8), (16, 8, 64, 0), (24, 32, 128, 16), (40, 16, 128, 4), (32, 8, 256, 5)])
def test_glm_epilogue_groups(R, most, n_r, n_c, d, n_co):
    # three groups of epilogue warps (two behind 40 embeddings of a request, or where a third takes a stage): runs of fewer
    # tiles than groups and runs that take each of them several times, with tiles that leave warps without rows
    co = wl.offsets_from_counts(np.random.default_rng(most).integers(0, most, R).tolist())
    cfg = wl.CONFIGS[5].with_(R=R, n_r=n_r, n_c=n_c, d_emb=d, n_ro=min(2, n_co), n_co=n_co)
    N = int(co[-1])
    sample = np.unique(np.concatenate([np.clip(np.stack([co[:-1], co[1:] - 1]).ravel(), 0, N - 1), np.arange(0, N, 61)]))
    assert _run_glm(cfg, co, sample=sample) <= tol_for("bf16")


def test_glm_config4_full_size_sampled():
    cfg = wl.CONFIGS[4]
    co = wl.cand_offsets(cfg)
    sample = wl.stratified_sample(co, n_uniform=512, n_small_requests=0, cfg_id=4)
    assert _run_glm(cfg, co, sample=sample) <= tol_for("bf16")


def test_glm_config5_full_size_sampled():
    cfg = wl.CONFIGS[5]
    co = wl.cand_offsets(cfg)
    sample = wl.stratified_sample(co, n_uniform=512, n_small_requests=8, cfg_id=5)
    assert _run_glm(cfg, co, sample=sample) <= tol_for("bf16")


# ------------------------------------------------------------------ isolation ---------------
def _bits(t):
    return t.contiguous().view(torch.uint8).cpu().numpy().reshape(t.shape[0], -1)


@pytest.mark.parametrize("path", PATHS)
def test_candidate_isolation_is_bit_exact(path):
    """Eq. 1 on the GPU: perturb one candidate, every other candidate's output bits stay put;
    perturb one request, only its own segment moves.  Also run-to-run determinism."""
    rocs.set_path(path)
    co = wl.offsets_from_counts([130, 1, 64, 300, 5, 150])
    so = wl.offsets_from_counts([150, 20, 128, 260, 64, 33])
    cfg = wl.CONFIGS[5].with_(R=6, d_req=128, d_cand=128, d_out=256, n_ro=4, n_co=4)
    plan = _plan(co)
    N = int(co[-1])
    j = int(co[3]) + 77           # a candidate in the middle of a tile
    seg = slice(int(co[2]), int(co[3]))

    lin = wl.linear_inputs(cfg, co)
    W, XR, XC = to_dev(lin["W"]), to_dev(lin["XR"]), to_dev(lin["XC"])
    att = wl.dca_inputs(cfg, co, so)
    Q, K, V, sod = to_dev(att["Q"]), to_dev(att["K"]), to_dev(att["V"]), to_dev(so)
    g = wl.glm_inputs(cfg, co)
    GR, GC, GW = to_dev(g["XR"]), to_dev(g["XC"]), to_dev(g["W"])

    def run_all(XR, XC, Q, K, GR, GC):
        y = rocs.ikbo_linear(plan, XR, XC, W[:, :cfg.d_req], W[:, cfg.d_req:], relu=True)
        o = rocs.dca_attention(plan, Q, K, V, sod)
        gi = rocs.glm_interaction(plan, GR, GC, GW, cfg.n_ro, cfg.n_co)
        return [_bits(y), _bits(o), _bits(gi["YC"]), _bits(gi["OC"])]

    base = run_all(XR, XC, Q, K, GR, GC)
    again = run_all(XR, XC, Q, K, GR, GC)
    for a, b in zip(base, again):
        assert np.array_equal(a, b), "not run-to-run deterministic"

    XC2, Q2, GC2 = XC.clone(), Q.clone(), GC.clone()
    XC2[j] += 1.0
    Q2[j] *= 1.5
    GC2[j] += 0.5
    pert = run_all(XR, XC2, Q2, K, GR, GC2)
    others = np.ones(N, bool)
    others[j] = False
    for a, b in zip(base, pert):
        assert np.array_equal(a[others], b[others]), "another candidate's output changed"
        assert not np.array_equal(a[j], b[j])

    XR2, K2, GR2 = XR.clone(), K.clone(), GR.clone()
    XR2[2] += 1.0
    K2[int(so[2]):int(so[3])] *= 0.5
    GR2[2] += 0.5
    pert = run_all(XR2, XC, Q, K2, GR2, GC)
    outside = np.ones(N, bool)
    outside[seg] = False
    for a, b in zip(base, pert):
        assert np.array_equal(a[outside], b[outside]), "a request leaked into another segment"
        assert np.all(np.any(a[seg] != b[seg], axis=1))


# ------------------------------------------------------------------ streams and graphs -------
@pytest.mark.parametrize("d_cand,d_out", [(128, 512), (320, 128)])   # candidate halves that release early and late
def test_threads_that_share_a_stream_have_request_tables_of_their_own(d_cand, d_out):
    # plans of different segments, made and dropped at once by each thread: the memory of one table is the next one's, and
    # other threads' launches come between a call's request half and its table
    g = np.random.default_rng(11)
    W = torch.randn((d_out, 64 + d_cand), device="cuda").to(torch.bfloat16)
    batches = []
    for R in (3, 40, 700, 2500):
        co = wl.offsets_from_counts(np.diff(np.sort(np.concatenate([[0, 20000], g.integers(0, 20001, R - 1)]))).tolist())
        XR, XC = torch.randn((R, 64), device="cuda").to(torch.bfloat16), torch.randn((20000, d_cand), device="cuda").to(torch.bfloat16)
        Z = XR.double() @ W[:, :64].double().T
        want = Z.repeat_interleave(to_dev(np.diff(co)), 0) + XC.double() @ W[:, 64:].double().T
        batches.append((to_dev(co), torch.from_numpy(co), XR, XC, want))
    torch.cuda.synchronize()

    def score(batch):
        cod, host, XR, XC, want = batch
        outs = []
        for _ in range(12):
            plan = rocs.plan_create(cod, host)
            outs.append(rocs.ikbo_linear(plan, XR, XC, W[:, :64], W[:, 64:]))
            plan.close()
        return max(float((y.double() - want).abs().max() / want.abs().max()) for y in outs)

    with ThreadPoolExecutor(len(batches)) as pool:
        for _ in range(4):
            assert max(pool.map(score, batches)) <= tol_for("bf16")


@pytest.mark.parametrize("warm", [False, True])
def test_calls_captured_in_a_graph_replay(warm):
    # a plan made outside the capture, used or not yet used when the capture begins; and a plan that lives inside the
    # capture.  Every call of this batch finds its work in the offsets; batches that need lists are below
    cfg = wl.CONFIGS[5].with_(R=5, d_req=64, d_cand=64, d_out=128, n_ro=4, n_co=4)
    co, so = wl.offsets_from_counts([30, 0, 700, 1, 9]), wl.offsets_from_counts([40, 10, 200, 5, 64])
    lin, att, g = wl.linear_inputs(cfg, co), wl.dca_inputs(cfg, co, so), wl.glm_inputs(cfg, co)
    W, XR, XC = to_dev(lin["W"]), to_dev(lin["XR"]), to_dev(lin["XC"])
    Q, K, V, sod = to_dev(att["Q"]), to_dev(att["K"]), to_dev(att["V"]), to_dev(so)
    GR, GC, GW = to_dev(g["XR"]), to_dev(g["XC"]), to_dev(g["W"])
    cod, host = to_dev(co), torch.from_numpy(co)

    def layers(plan):
        y = rocs.ikbo_linear(plan, XR, XC, W[:, :cfg.d_req], W[:, cfg.d_req:], relu=True)
        o = rocs.dca_attention(plan, Q, K, V, sod)
        return [y, o, rocs.glm_interaction(plan, GR, GC, GW, cfg.n_ro, cfg.n_co)["OC"]]

    other = rocs.plan_create(cod, host)
    want = [_bits(t) for t in layers(other)]
    plan = other if warm else rocs.plan_create(cod, host)
    for inside in (False, True):
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            p = rocs.plan_create(cod, host) if inside else plan
            outs = layers(p)
            if inside:
                p.close()
        for _ in range(3):
            for t in outs:
                t.zero_()
            graph.replay()
            assert all(np.array_equal(_bits(t), w) for t, w in zip(outs, want))
    again = layers(plan)   # and the plan still serves calls outside the graph
    assert all(np.array_equal(_bits(t), w) for t, w in zip(again, want))


def _lists(plan, captured=False):
    fn = rocs.lib().rocs_selftest_plan_lists
    fn.argtypes = [ctypes.c_void_p, ctypes.c_int]
    return fn(plan.handle, int(captured))


class _ListedBatch:
    """A batch whose calls all need a list of the plan: the request table of more than 16384 candidates, the attention
    items of more than 256 requests (fp32: 128) and the interaction tiles of more than 512 (fp32: 128)."""
    LISTS = 5   # one for bf16 linear, attention and interaction each, two for the fp32 ones

    def __init__(self):
        g = np.random.default_rng(4)
        self.co = wl.offsets_from_counts(g.integers(0, 68, 600).tolist())
        so = wl.offsets_from_counts(g.integers(1, 40, 600).tolist())
        cfg = wl.CONFIGS[5].with_(R=600, d_req=64, d_cand=64, d_out=128, H=2, dh=32, n_r=8, n_c=8, d_emb=64, n_ro=4, n_co=4)
        assert int(self.co[-1]) > 16384
        lin, att, gi = wl.linear_inputs(cfg, self.co), wl.dca_inputs(cfg, self.co, so), wl.glm_inputs(cfg, self.co)
        self.W, self.XR, self.XC = to_dev(lin["W"]), to_dev(lin["XR"]), to_dev(lin["XC"])
        self.Q, self.K, self.V, self.so = to_dev(att["Q"]), to_dev(att["K"]), to_dev(att["V"]), to_dev(so)
        self.GR, self.GC, self.GW = to_dev(gi["XR"]), to_dev(gi["XC"]), to_dev(gi["W"])
        self.f = [t.float() for t in (self.Q, self.K, self.V, self.GR, self.GC)]
        self.cod, self.host = to_dev(self.co), torch.from_numpy(self.co)
        torch.cuda.synchronize()

    def plan(self):
        return rocs.plan_create(self.cod, self.host)

    def layers(self, plan):
        Q, K, V, GR, GC = self.f
        return [rocs.ikbo_linear(plan, self.XR, self.XC, self.W[:, :64], self.W[:, 64:], relu=True),
                rocs.dca_attention(plan, self.Q, self.K, self.V, self.so),
                rocs.glm_interaction(plan, self.GR, self.GC, self.GW, 4, 4)["OC"],
                rocs.dca_attention(plan, Q, K, V, self.so),
                rocs.glm_interaction(plan, GR, GC, None)["YC"]]


def _same(outs, want):
    return all(np.array_equal(_bits(t), w) for t, w in zip(outs, want))


@pytest.mark.parametrize("before", ["nothing", "plan's stream", "another stream"])
def test_captured_calls_find_lists_made_outside(before):
    # what the plan holds when the capture begins: nothing, lists made on its stream (the graph may read them), lists made
    # on a stream that the graph's is not ordered behind (it must not)
    b = _ListedBatch()
    want = [_bits(t) for t in b.layers(b.plan())]
    plan = b.plan()
    if before == "plan's stream":
        b.layers(plan)
    elif before == "another stream":
        with torch.cuda.stream(torch.cuda.Stream()):
            b.layers(plan)
    had = _lists(plan)
    assert had == (0 if before == "nothing" else b.LISTS)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        outs = b.layers(plan)
    assert _lists(plan) == had + (0 if before == "plan's stream" else b.LISTS)
    for _ in range(3):
        for t in outs:
            t.zero_()
        graph.replay()
        assert _same(outs, want)
    assert _same(b.layers(plan), want)     # what was complete when it was made serves eager calls too
    assert _lists(plan) == had + (0 if before == "plan's stream" else b.LISTS)


@pytest.mark.parametrize("closed_inside", [True, False])
def test_a_plan_created_inside_a_capture(closed_inside):
    # its lists are the graph's memory; eager calls on it, if it stays open, make lists of their own
    b = _ListedBatch()
    want = [_bits(t) for t in b.layers(b.plan())]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        plan = b.plan()
        outs = b.layers(plan)
        assert _lists(plan) == 0 and _lists(plan, captured=True) == b.LISTS
        if closed_inside:
            plan.close()
    if not closed_inside:
        assert _same(b.layers(plan), want)
        assert _lists(plan) == b.LISTS
    for _ in range(3 if closed_inside else 1):
        for t in outs:
            t.zero_()
        graph.replay()
        assert _same(outs, want)
    if not closed_inside:
        assert _same(b.layers(plan), want)
        torch.cuda.synchronize()
        plan.close()
    assert rocs.last_device_status() == 0


def test_a_graph_of_more_requests_than_a_block_adds_up_keeps_nothing_of_the_host():
    # the plan lives inside the capture and its lists are made at every replay, when the calls' host memory is long reused
    R = 12001
    g = np.random.default_rng(9)
    co, so = wl.offsets_from_counts(g.integers(0, 4, R).tolist()), wl.offsets_from_counts(g.integers(0, 5, R).tolist())
    cfg = wl.CONFIGS[5].with_(R=R, H=2, dh=32, n_r=8, n_c=8, d_emb=64, n_ro=0, n_co=0)
    att, gi = wl.dca_inputs(cfg, co, so), wl.glm_inputs(cfg, co)
    Q, K, V, sod, GR, GC = (to_dev(a) for a in (att["Q"], att["K"], att["V"], so, gi["XR"], gi["XC"]))
    cod, host = to_dev(co), torch.from_numpy(co)

    def layers(plan):
        return [rocs.dca_attention(plan, Q, K, V, sod), rocs.glm_interaction(plan, GR, GC, None)["YC"]]

    want = [_bits(t) for t in layers(rocs.plan_create(cod, host))]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        plan = rocs.plan_create(cod, host)
        outs = layers(plan)
        plan.close()
    for _ in range(3):
        junk = [np.full(R + 1, 7, np.int32) for _ in range(200)]
        for t in outs:
            t.zero_()
        graph.replay()
        assert _same(outs, want)
        del junk


def test_calls_on_a_kept_plan_do_not_walk_its_requests():
    # the host's share of a call (it returns without waiting for the device) on 200000 requests: a walk over the offsets is
    # some 180 us, and an interaction took two; without, a call is some 10 us
    R = 200000
    co = torch.arange(R + 1, dtype=torch.int32)
    so = torch.arange(R + 1, dtype=torch.int32, device="cuda")
    bf = dict(dtype=torch.bfloat16, device="cuda")
    XR, XC, Q = torch.zeros((R, 8, 64), **bf), torch.zeros((R, 8, 64), **bf), torch.zeros((R, 1, 1, 32), **bf)
    plan = rocs.plan_create(co.cuda(), co)
    raw, att = {"YC": torch.empty((R, 8, 16), **bf)}, torch.empty_like(Q)
    calls = {"interaction": lambda: rocs.glm_interaction(plan, XR, XC, None, want_request_side=False, outs=raw),
             "attention": lambda: rocs.dca_attention(plan, Q, Q[:, 0], Q[:, 0], so, out=att)}
    for name, call in calls.items():
        took = []
        for _ in range(21):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            call()
            took.append(time.perf_counter() - t0)
        assert sorted(took)[10] < 150e-6, (name, sorted(took)[10])
    torch.cuda.synchronize()


def test_no_item_of_a_split_batch_waits_for_a_second_round():
    # 16 items of which not every one gets a cluster at the same time take nearly twice as long as 14 that do
    bf = dict(device="cuda", dtype=torch.bfloat16)

    def took(R, H, L=4096):
        co = torch.arange(0, R * 50 + 1, 50, dtype=torch.int32)
        so = torch.arange(0, R * L + 1, L, dtype=torch.int32, device="cuda")
        Q, K, V = torch.zeros((R * 50, 1, H, 64), **bf), torch.zeros((R * L, H, 64), **bf), torch.zeros((R * L, H, 64), **bf)
        plan, out = rocs.plan_create(co.cuda(), co), torch.empty_like(Q)
        a, b, times = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True), []
        for _ in range(6):
            a.record()
            for _ in range(50):
                rocs.dca_attention(plan, Q, K, V, so, out=out)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)

    assert took(2, 8) < 1.4 * took(2, 7)


def test_one_plan_on_two_streams():
    # lists of either stream's own, made at the same time; results are those of one stream
    b = _ListedBatch()
    want = [_bits(t) for t in b.layers(b.plan())]
    plan, streams = b.plan(), [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    outs = []
    for _ in range(4):
        for s in streams:
            with torch.cuda.stream(s):
                outs.append(b.layers(plan))
    torch.cuda.synchronize()
    assert _lists(plan) == 2 * b.LISTS
    assert all(_same(o, want) for o in outs)


# ------------------------------------------------------------------ ABI errors --------------
def test_outputs_that_are_lazy_clones_leave_their_source_alone():
    co = wl.offsets_from_counts([3, 5])
    plan = _plan(co)
    def t(*shape):
        return torch.randn(shape, device="cuda").to(torch.bfloat16)
    source = torch.full((8 * 64,), 7.0, dtype=torch.bfloat16, device="cuda")
    def out(*shape):
        return torch._lazy_clone(source)[:int(np.prod(shape))].view(shape)
    W, stats = t(64, 64), torch._lazy_clone(torch.zeros((8, 2), device="cuda"))
    rocs.linear(t(8, 64), W, out=out(8, 64))
    rocs.ikbo_linear(plan, t(2, 64), t(8, 64), W, W, out=out(8, 64))
    rocs.ikbo_linear_stats(plan, t(2, 64), t(8, 64), W, W, out=out(8, 64), row_stats=stats)
    rocs.ikbo_linear_static(to_dev(co), t(2, 64), t(8, 64), W, W, out(8, 64))
    rocs.group_norm(t(8, 64), out=out(8, 64))
    rocs.dca_attention(plan, t(8, 1, 2, 32), t(6, 2, 32), t(6, 2, 32), to_dev(np.array([0, 4, 6], np.int32)), out=out(8, 1, 2, 32))
    rocs.glm_interaction(plan, t(2, 2, 64), t(8, 2, 64), None, outs={"YR": out(2, 2, 4), "YC": out(8, 2, 4)})
    rocs.glm_fm_projection(plan, t(2, 2, 64), t(8, 2, 64), t(4, 8), outs={"FR": out(2, 2, 8), "FC": out(8, 2, 8)})
    assert bool((source == 7.0).all())


def test_an_output_that_does_not_fit_raises_torchs_own_error():
    X = torch.zeros((1, 64), dtype=torch.bfloat16, device="cuda").expand(1 << 31, 64)
    W = torch.zeros((4096, 64), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(torch.OutOfMemoryError):
        rocs.linear(X, W)


def test_error_codes_on_bad_arguments():
    co = wl.offsets_from_counts([4, 4])
    d_co = to_dev(co)
    with pytest.raises(rocs.RocsError) as e:
        rocs.plan_create(d_co, np.array([0, 5, 4], np.int32))
    assert e.value.code == -4
    with pytest.raises(rocs.RocsError) as e:
        rocs.plan_create(d_co, np.array([1, 4, 8], np.int32))
    assert e.value.code == -4
    plan = rocs.plan_create(d_co)                # host copy omitted: read back from the device
    assert plan.N == 8
    X = torch.zeros((8, 72), dtype=torch.bfloat16, device="cuda")
    XR = torch.zeros((2, 64), dtype=torch.bfloat16, device="cuda")
    W = torch.zeros((16, 136), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(rocs.RocsError) as e:     # misaligned view: column offset of 2 bytes
        rocs.ikbo_linear(plan, XR, X[:, 1:65], W[:, :64], W[:, 64:128])
    assert e.value.code == -2
    with pytest.raises(rocs.RocsError) as e:     # workspace too small
        rocs.ikbo_linear(plan, XR, X[:, :64], W[:, :64], W[:, 64:128],
                         workspace=torch.empty(16, dtype=torch.uint8, device="cuda"))
    assert e.value.code == -5
    Q = torch.zeros((8, 1, 2, 36), dtype=torch.bfloat16, device="cuda")
    KV = torch.zeros((6, 2, 36), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(rocs.RocsError) as e:     # dh * 2 bytes not a multiple of 16
        rocs.dca_attention(plan, Q, KV, KV, to_dev(np.array([0, 3, 6], np.int32)))
    assert e.value.code == -2
