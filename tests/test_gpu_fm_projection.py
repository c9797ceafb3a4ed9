"""GPU parity of the projected factorization machine (F = G P on Eq. 9-10) against the fp64 oracle,
through the C ABI.  bf16: max |gpu - ref| <= 1e-2 max |ref|; fp32: 1e-4; isolation: bit-exact."""
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


def _run(cfg, co, k, sample=None, path=rocs.PATH_AUTO):
    rocs.set_path(path)
    d = wl.glm_inputs(cfg, co)
    P = wl.fm_projection_weight(cfg, k)
    plan = rocs.plan_create(to_dev(co), co)
    outs = rocs.glm_fm_projection(plan, to_dev(d["XR"]), to_dev(d["XC"]), to_dev(P))
    F = ref.glm_fm_projection(co, d["XR"], d["XC"], P, sample=sample)
    if F.shape[0] == 0:
        return 0.0
    m = np.repeat(np.arange(cfg.R), np.diff(co))
    sel = (lambda a: a) if sample is None else (lambda a: a[sample])
    return max(rel_err(sel(to_host_f64(outs["FC"])), F[:, cfg.n_r:]),
               rel_err(sel(to_host_f64(outs["FR"])[m]), F[:, :cfg.n_r]))


def test_config1_fp32_every_element():
    cfg = wl.CONFIGS[1]
    assert _run(cfg, wl.cand_offsets(cfg), k=5) <= tol_for("f32")


@pytest.mark.parametrize("path", PATHS)
@pytest.mark.parametrize("k", [8, 16])
@pytest.mark.parametrize("d_emb", [64, 128, 192, 256])
def test_bf16_ragged_segments_and_tail_tile(path, k, d_emb):
    # empty requests, single candidates, segments that straddle the 8-candidate tiles, N % 8 != 0
    co = wl.offsets_from_counts([1, 0, 9, 8, 33, 7, 0, 133])
    cfg = wl.CONFIGS[4].with_(R=len(co) - 1, d_emb=d_emb)
    assert _run(cfg, co, k, path=path) <= tol_for("bf16")


@pytest.mark.parametrize("n_c,k", [(16, 8), (16, 16), (12, 8), (4, 8)])
@pytest.mark.parametrize("law", ["short", "gaps", "long"])
def test_bf16_streaming_kernel_walks_the_requests(law, n_c, k):
    # a warp's candidates ascend by 8 or 15, in several tiles per CTA: the next request, the one behind a run of empty ones, the same
    # one (4 embeddings: by more than two candidates per tile the walk over tiles of the tcgen05 kernel)
    g = np.random.default_rng(5)
    counts = {"short": g.integers(0, 4, 9000), "gaps": np.where(g.random(9000) < 0.02, g.integers(1, 150, 9000), 0),
              "long": g.integers(500, 3000, 9)}[law]
    co = wl.offsets_from_counts(counts.tolist())
    cfg = wl.CONFIGS[4].with_(R=len(co) - 1, n_r=4, n_c=n_c, d_emb=64)
    sample = np.unique(np.concatenate([g.integers(0, co[-1], 600), [0, co[-1] - 1]]))
    assert _run(cfg, co, k, sample=sample) <= tol_for("bf16")


@pytest.mark.parametrize("n_c,k,d_emb", [(12, 16, 128), (4, 24, 192), (1, 2, 64), (15, 32, 256), (16, 18, 128), (8, 10, 64)])
def test_bf16_streaming_kernel_with_partial_fragments(n_c, k, d_emb):
    # fewer than 16 rows per candidate (fragments reach into the next candidate's rows), one and two blocks of
    # projection columns, the last of them partial; a candidate full of NaN must not show in its neighbours
    co = wl.offsets_from_counts([1, 0, 9, 8, 33, 7, 0, 133])
    cfg = wl.CONFIGS[4].with_(R=len(co) - 1, n_r=20, n_c=n_c, d_emb=d_emb)
    assert _run(cfg, co, k) <= tol_for("bf16")
    d = wl.glm_inputs(cfg, co)
    P, XC = to_dev(wl.fm_projection_weight(cfg, k)), to_dev(d["XC"])
    plan = rocs.plan_create(to_dev(co), co)
    base = _bits(rocs.glm_fm_projection(plan, to_dev(d["XR"]), XC, P)["FC"])
    XC[60] = float("nan")
    pert = _bits(rocs.glm_fm_projection(plan, to_dev(d["XR"]), XC, P)["FC"])
    others = np.arange(len(base)) != 60
    assert np.array_equal(base[others], pert[others])


@pytest.mark.parametrize("n_c,k,d_emb", [(12, 16, 128), (4, 24, 192), (15, 32, 256), (16, 18, 128), (16, 12, 64), (8, 8, 64)])
@pytest.mark.parametrize("counts", [[1, 0, 9, 8, 33, 7, 0, 133], [1, 0, 2] * 70])
def test_bf16_partial_fragments_are_as_exact_as_fp32_arithmetic(n_c, k, d_emb, counts):
    # Both kernels hold T and the candidate's own term to fp32 and round the result to bf16 once.  Sums of fp32 in another order differ by some 2^-20,
    # against the 2^-9 of that rounding: the errors against fp64 are the same up to which way close values are rounded
    # (well below 1 % of the norm over these thousands of values; H in bf16 would add about 40 %).
    co = wl.offsets_from_counts(counts)  # (short requests are the streaming kernel's)
    cfg = wl.CONFIGS[4].with_(R=len(co) - 1, n_r=20, n_c=n_c, d_emb=d_emb)
    d, P = wl.glm_inputs(cfg, co), wl.fm_projection_weight(cfg, k)
    want = ref.glm_fm_projection(co, d["XR"], d["XC"], P)[:, cfg.n_r:]
    plan = rocs.plan_create(to_dev(co), co)
    XC = d["XC"].copy()
    XC[60, 1, 5] = 0x7f80   # and an infinity shows in the same values either way
    err, kinds = [], []
    for path in PATHS:
        rocs.set_path(path)
        got = to_host_f64(rocs.glm_fm_projection(plan, to_dev(d["XR"]), to_dev(d["XC"]), to_dev(P))["FC"])
        err.append(np.linalg.norm(got - want) / np.linalg.norm(want))
        got = to_host_f64(rocs.glm_fm_projection(plan, to_dev(d["XR"]), to_dev(XC), to_dev(P))["FC"])
        kinds.append(np.where(np.isnan(got), 2, np.where(np.isinf(got), np.sign(got), 0)))
    assert err[0] <= 1.01 * err[1]
    assert np.array_equal(kinds[0], kinds[1]) and np.any(kinds[1][60] != 0)


@pytest.mark.parametrize("law", ["few", "many", "sparse", "short"])
@pytest.mark.parametrize("n_r,n_c,d_emb,k", [(20, 12, 128, 16), (5, 3, 64, 2), (24, 4, 192, 24), (16, 5, 64, 14), (48, 8, 256, 32), (7, 9, 128, 22),
                                             (20, 16, 64, 24), (33, 15, 192, 8), (16, 1, 128, 16)])
def test_bf16_tiles_of_one_request(n_r, n_c, d_emb, k, law):
    # tiles of 8 to 32 candidates of one request, rows behind a candidate's embeddings and columns behind k; fewer tiles than a
    # ring has stages and runs that take ring and accumulators several times; more requests than threads, most of them empty;
    # a candidate or two per request, which the streaming kernel takes
    g = np.random.default_rng(k)
    counts = {"few": [3, 0, 33, 1], "many": g.integers(0, 130, 300), "sparse": np.where(g.random(3000) < 0.2, g.integers(1, 40, 3000), 0),
              "short": g.integers(0, 3, 600)}[law]
    co = wl.offsets_from_counts(np.asarray(counts).tolist())
    cfg = wl.CONFIGS[4].with_(R=len(co) - 1, n_r=n_r, n_c=n_c, d_emb=d_emb)
    N = int(co[-1])
    sample = np.unique(np.concatenate([g.integers(0, N, 400), [0, N - 1]]))
    assert _run(cfg, co, k, sample=sample) <= tol_for("bf16")
def _bf16(a):
    return torch.from_numpy(np.asarray(a, np.float32)).bfloat16()


def _error_by_path(co, XR, XC, P):
    """Relative error (2-norm) of FC against 64 bits on either path, and the 64-bit values."""
    want = ref.glm_fm_projection(co, *[t.view(torch.uint16).numpy() for t in (XR, XC, P)])[:, XR.shape[1]:]
    plan = rocs.plan_create(to_dev(co), co)
    err = []
    for path in PATHS:
        rocs.set_path(path)
        got = to_host_f64(rocs.glm_fm_projection(plan, XR.cuda(), XC.cuda(), P.cuda())["FC"])
        err.append(np.linalg.norm(got - want) / np.linalg.norm(want))
    return err, want


@pytest.mark.parametrize("n_c,k,d_emb", [(12, 16, 128), (4, 24, 192), (15, 32, 256), (8, 8, 128), (5, 2, 192)])
def test_bf16_request_term_keeps_its_24_bits(n_c, k, d_emb):
    # T is M + M / 256 + delta, delta some 2^-14, and neighbouring values of the candidates cancel what the first two give: FC is
    # X^C delta.  fp32 holds T to 2^-24 (2^-23 where a product's sum is cut off and not rounded), 2^-9 of delta at most; 17 bits
    # to 2^-18, 4 % of FC.
    g = np.random.default_rng(k)
    co = wl.offsets_from_counts([4000, 0, 3, 2500])  # as many tiles as the tcgen05 kernel is taken for
    R, N = len(co) - 1, int(co[-1])
    M = np.repeat(1.0 + g.random((R, 2, d_emb // 2)), 2, axis=2) * np.array([[1.0], [2.0 ** -8]])
    XR = _bf16(np.concatenate([M, 2.0 ** -14 * g.standard_normal((R, 1, d_emb))], axis=1))
    half = g.standard_normal((N, n_c, d_emb // 2, 1))
    XC = _bf16(np.concatenate([half, -half], axis=3).reshape(N, n_c, d_emb))
    P = _bf16(np.concatenate([np.ones((3, k)), 2.0 ** -30 * g.standard_normal((n_c, k))]))
    err, _ = _error_by_path(co, XR, XC, P)
    assert err[1] <= 3e-3 and err[0] <= (1.01 * err[1] ** 2 + 2.0 ** -18) ** 0.5, err


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -70])
@pytest.mark.parametrize("n_c,k,d_emb", [(12, 16, 128), (4, 24, 192), (15, 32, 256), (8, 8, 128), (5, 2, 192)])
def test_bf16_terms_that_cancel(n_c, k, d_emb, scale):
    # The candidates are small changes of their request's rows, and P_R = -P_C: X^C T and (X^C X^C^T) P_C are thousands of times
    # their sum, and would be off by up to a few 1e-3 of it as sums of their own.  Rows whose sum is below a 256th of a term are added
    # up before the product; what the others lose (256 times some 2^-21) is a sixteenth of FC's rounding, 2^-8 of it in the norm.
    # Scaled, the squares lie below fp32's range, and their products with P_C do not.
    g = np.random.default_rng(n_c)
    co = wl.offsets_from_counts([7000, 0, 3, 90])
    base = _bf16(g.standard_normal((4, n_c, d_emb))).double().numpy()
    PC = _bf16(g.standard_normal((n_c, k)) / n_c ** 0.5).double().numpy()
    X = np.repeat(base, np.diff(co), axis=0)
    at = g.integers(0, n_c * d_emb, (len(X), 4))
    np.put_along_axis(X.reshape(len(X), -1), at, np.take_along_axis(X.reshape(len(X), -1), at, 1) * (1 + 2.0 ** -6), 1)
    X = _bf16(X).double().numpy()
    err, _ = _error_by_path(co, _bf16(base * scale), _bf16(X * scale), _bf16(np.concatenate([-PC, PC]) / scale))
    assert err[1] <= 2e-3 and err[0] <= 1.01 * err[1], err


@pytest.mark.parametrize("where", ["XR nan", "XR inf", "XC nan", "XC inf", "P request nan", "P candidate inf", "XC huge"])
@pytest.mark.parametrize("n_c,k,d_emb", [(12, 16, 128), (4, 24, 192), (16, 20, 128), (8, 10, 128), (15, 32, 256)])
def test_bf16_values_out_of_range_show_as_in_fp32(n_c, k, d_emb, where):
    # NaN, infinity and squares past fp32 in some rows of a batch of many tiles: the same values are NaN or infinite as on the
    # general path, and the others' bits do not change
    g = np.random.default_rng(n_c)
    co = wl.offsets_from_counts(g.integers(0, 100, 130).tolist())
    cfg = wl.CONFIGS[4].with_(R=len(co) - 1, n_r=20, n_c=n_c, d_emb=d_emb)
    d = wl.glm_inputs(cfg, co)
    d["P"] = wl.fm_projection_weight(cfg, k)
    plan = rocs.plan_create(to_dev(co), co)
    run = lambda: rocs.glm_fm_projection(plan, *[to_dev(d[n]) for n in ("XR", "XC", "P")])["FC"]
    before = _bits(run())
    bits = {"nan": 0x7fc0, "inf": 0x7f80, "huge": 0x6500}[where.split()[-1]]
    if where.startswith("P"):
        d["P"][3 if "request" in where else 20 + n_c - 1, k // 2] = bits
        touched = np.ones(len(before), bool)
    elif where.startswith("XR"):
        d["XR"][[5, 77], [2, 19], [7, 63]] = bits
        touched = np.isin(np.repeat(np.arange(cfg.R), np.diff(co)), [5, 77])
    else:
        rows = [0, 33, 34, len(before) - 1]
        d["XC"][rows, [0, n_c - 1, 1, 2], [1, 0, d_emb - 1, 5]] = bits
        touched = np.isin(np.arange(len(before)), rows)
    kinds, got = [], None
    for path in PATHS:
        rocs.set_path(path)
        out = run()
        got = _bits(out) if got is None else got
        out = to_host_f64(out)
        kinds.append(np.where(np.isnan(out), 2, np.where(np.isinf(out), np.sign(out), 0)))
    assert np.array_equal(kinds[0], kinds[1])
    assert np.any(kinds[1][touched] != 0) or where == "XC huge"
    assert np.array_equal(got[~touched], before[~touched])


@pytest.mark.parametrize("path", PATHS)
def test_bf16_shapes_outside_the_streaming_kernel(path):
    co = wl.offsets_from_counts([20, 3, 41])
    cfg = wl.CONFIGS[4].with_(R=3, n_r=24, n_c=8, d_emb=64)
    assert _run(cfg, co, 12, path=path) <= tol_for("bf16")
    cfg = wl.CONFIGS[4].with_(R=3, n_r=8, n_c=16, d_emb=32)
    assert _run(cfg, co, 16, path=path) <= tol_for("bf16")


def test_wide_request_group():
    co = wl.offsets_from_counts([3, 70, 5])
    cfg = wl.CONFIGS[4].with_(R=3, n_r=64, d_emb=256)
    assert _run(cfg, co, 16) <= tol_for("bf16")


def test_many_tiles_per_cta():
    # more tiles than CTAs: every CTA goes around its ring several times and changes request mid-run
    g = np.random.default_rng(7)
    co = wl.offsets_from_counts(g.integers(0, 200, size=120).tolist())
    cfg = wl.CONFIGS[4].with_(R=len(co) - 1)
    assert _run(cfg, co, 16) <= tol_for("bf16")


def test_config4_full_size_sampled():
    cfg = wl.CONFIGS[4]
    co = wl.cand_offsets(cfg)
    sample = wl.stratified_sample(co, n_uniform=512, n_small_requests=0, cfg_id=4)
    assert _run(cfg, co, 16, sample=sample) <= tol_for("bf16")


def _bits(t):
    return t.contiguous().view(torch.uint8).cpu().numpy().reshape(t.shape[0], -1)


@pytest.mark.parametrize("path", PATHS)
def test_candidate_isolation_is_bit_exact(path):
    rocs.set_path(path)
    co = wl.offsets_from_counts([130, 1, 64, 300, 5, 150])
    cfg = wl.CONFIGS[4].with_(R=6)
    d = wl.glm_inputs(cfg, co)
    P = to_dev(wl.fm_projection_weight(cfg, 16))
    plan = rocs.plan_create(to_dev(co), co)
    XR, XC = to_dev(d["XR"]), to_dev(d["XC"])
    N = int(co[-1])
    j = int(co[3]) + 77
    seg = slice(int(co[2]), int(co[3]))
    base = _bits(rocs.glm_fm_projection(plan, XR, XC, P)["FC"])
    assert np.array_equal(base, _bits(rocs.glm_fm_projection(plan, XR, XC, P)["FC"])), "not deterministic"
    XC2 = XC.clone()
    XC2[j] += 0.5
    pert = _bits(rocs.glm_fm_projection(plan, XR, XC2, P)["FC"])
    others = np.ones(N, bool)
    others[j] = False
    assert np.array_equal(base[others], pert[others]) and not np.array_equal(base[j], pert[j])
    XR2 = XR.clone()
    XR2[2] += 0.5
    pert = _bits(rocs.glm_fm_projection(plan, XR2, XC, P)["FC"])
    outside = np.ones(N, bool)
    outside[seg] = False
    assert np.array_equal(base[outside], pert[outside]), "a request leaked into another segment"
    assert np.all(np.any(base[seg] != pert[seg], axis=1))


def test_error_codes():
    co = wl.offsets_from_counts([4, 4])
    cfg = wl.CONFIGS[4].with_(R=2)
    d = wl.glm_inputs(cfg, co)
    plan = rocs.plan_create(to_dev(co), co)
    XR, XC, P = to_dev(d["XR"]), to_dev(d["XC"]), to_dev(wl.fm_projection_weight(cfg, 16))
    with pytest.raises(rocs.RocsError) as e:
        rocs.glm_fm_projection(plan, XR, XC, P, workspace=torch.empty(16, dtype=torch.uint8, device="cuda"))
    assert e.value.code == -5  # ROCS_ERR_WORKSPACE
    need = rocs.glm_fm_projection_workspace(plan, cfg.d_emb, 16)
    assert need >= 2 * 16 * cfg.d_emb * 4 and need % 256 == 0
