"""Attention layer (Heterogeneous Graph Transformer, Eq. 6-11) forward and backward through the C
ABI against the oracle, on seeded power-law graphs whose in- and out-degree hubs exceed the hub
degree (so the chunked paths of all three edge passes run), ragged type sizes and isolated nodes."""
from types import SimpleNamespace

import numpy as np
import pytest
import torch

import hgsynth
from oracle import hgt as OH
from tests.gpu_util import BF16_RELU_MARGIN, TOL, dev, host, lib, need_gpu, relerr, tdtype

pytestmark = pytest.mark.gpu

KEYS = ("W_K", "W_Q", "W_V", "b_K", "b_Q", "b_V", "W_att", "W_msg", "mu", "W_agg", "b_agg", "ln_gamma", "ln_beta")

CASES = {
    "tiny-f32-d64-h4": ("tiny-10k", {}, 4),
    "sub-bf16-d128-h4": ("sub-1m", dict(n_user=27_001, n_risk=3_003, num_edges=600_000, n_overlap=4_000), 4),
    "tiny-bf16-d64-h8": ("tiny-10k", dict(dtype="bf16"), 8),
    "sub-f32-d128-h1": ("sub-1m", dict(n_user=9_001, n_risk=1_003, num_edges=150_000, n_overlap=1_000, dtype="f32"), 1),
    "tail-bf16-d256-h4": ("tail-5m", dict(n_user=9_007, n_risk=1_001, num_edges=200_000, n_overlap=1_000,
                                          out_cap=4_000), 4),
}


def run_gpu(hg, w, p, heads, ln, dOut):
    sp, g = w.spec, w.graph
    td = tdtype(sp.dtype)
    G = hg.hg_build_csr(dev(g["src"]), dev(g["dst"]), dev(g["rel"]), g["type_offsets"], g["rels"])
    tens = {k: dev(p[k], torch.float32 if k == "mu" else td) for k in KEYS}
    P = hg.HgtParams(tens, heads, layernorm=ln)
    sb, kb = hg.hg_hgt_workspace_size(G, P)
    saved = torch.empty(sb, dtype=torch.uint8, device="cuda")
    scratch = torch.empty(kb, dtype=torch.uint8, device="cuda")
    X = dev(w.X, td)
    out = torch.empty_like(X)
    hg.hg_hgt_fwd(G, P, X, out, saved, scratch)
    dH = torch.empty_like(X)
    grads = {k: torch.full(np.shape(p[k]), np.nan, dtype=torch.float32, device="cuda") for k in KEYS}
    hg.hg_hgt_bwd(G, P, X, saved, dev(dOut, td), dH, grads, scratch)
    torch.cuda.synchronize()
    return host(out), host(dH), {k: host(v) for k, v in grads.items()}


@pytest.mark.parametrize("case", list(CASES))
@pytest.mark.parametrize("ln", [True, False])
def test_hgt_matches_oracle(case, ln):
    need_gpu()
    hg = lib()
    name, ov, heads = CASES[case]
    sp = hgsynth.spec(name, **ov)
    # bf16 ReLU: biases of +-8 keep the pre-activations clear of the kink (as for the mean layer)
    w = hgsynth.make_workload(sp, random_affine=True, with_ids=False)
    p = hgsynth.make_hgt_params(sp, heads, bias_margin=BF16_RELU_MARGIN if sp.dtype == "bf16" else None)
    g = w.graph
    out, dH, gr = run_gpu(hg, w, p, heads, ln, w.dH_top)
    args = (g["src"], g["dst"], g["rel"], g["type_offsets"], g["rels"], p, w.X)
    ref, _ = OH.hgt_forward(*args, heads, layernorm=ln)  # the plain fp64 definition (Eq. 6-11)
    tol = TOL[sp.dtype]
    assert relerr(out, ref) <= tol, ("H_out", relerr(out, ref))
    dref, gref = OH.hgt_backward(*args, w.dH_top, heads, layernorm=ln)
    assert relerr(dH, dref) <= tol, ("dH_in", relerr(dH, dref))
    for k in KEYS:
        if not ln and k in ("ln_gamma", "ln_beta"):
            continue
        e = relerr(gr[k], gref[k])
        assert e <= tol, (k, e)
    assert hg.hg_device_status() == 0


def test_hgt_is_bitwise_repeatable():
    need_gpu()
    hg = lib()
    name, ov, heads = CASES["sub-bf16-d128-h4"]
    sp = hgsynth.spec(name, **ov)
    w = hgsynth.make_workload(sp, random_affine=True, with_ids=False)
    p = hgsynth.make_hgt_params(sp, heads)
    a = run_gpu(hg, w, p, heads, True, w.dH_top)
    b = run_gpu(hg, w, p, heads, True, w.dH_top)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    for k in KEYS:
        assert np.array_equal(a[2][k], b[2][k]), k


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("rows", [1, 128, 129])
def test_hgt_few_stored_rows(dtype, rows):
    """Only `rows` targets of relation 0 have in-edges and relation 1 has none: products over the stored rows at the
    edges of a 128-row tile, and over no rows at all."""
    need_gpu()
    hg = lib()
    sp = hgsynth.spec("tiny-10k", n_user=401, n_risk=103, num_edges=6_000, n_overlap=10, dtype=dtype)
    w = hgsynth.make_workload(sp, random_affine=True, with_ids=False)
    p = hgsynth.make_hgt_params(sp, 4, bias_margin=BF16_RELU_MARGIN if dtype == "bf16" else None)
    g = w.graph
    keep = np.flatnonzero(g["rel"] == 0)
    for k in ("src", "dst", "rel"):
        g[k] = np.ascontiguousarray(g[k][keep])
    lo = g["type_offsets"][g["rels"][0][1]]
    g["dst"] = (lo + np.arange(keep.size) % rows).astype(g["dst"].dtype)
    out, dH, gr = run_gpu(hg, w, p, 4, True, w.dH_top)
    args = (g["src"], g["dst"], g["rel"], g["type_offsets"], g["rels"], p, w.X)
    ref, _ = OH.hgt_forward(*args, 4, layernorm=True)
    dref, gref = OH.hgt_backward(*args, w.dH_top, 4, layernorm=True)
    assert relerr(out, ref) <= TOL[dtype] and relerr(dH, dref) <= TOL[dtype]
    for k in KEYS:
        # with one relation b_K shifts all scores of a softmax alike: its gradient is zero, what is left is rounding;
        # dmu = <W_att, dW_att> / mu, a sum of cancelling terms, is off by at most |W_att| |error of dW_att| / mu
        scale = np.abs(gref["W_K" if k == "b_K" else k]).max()
        if k == "mu":
            scale = np.linalg.norm(p["W_att"][0]) * np.linalg.norm(gref["W_att"][0]) / abs(p["mu"][0])
        assert np.abs(gr[k] - gref[k]).max() <= TOL[dtype] * scale, k
    assert hg.hg_device_status() == 0


def test_scores_of_minus_infinity():
    """Parts of a row whose scores all overflow to -inf: the first four runs of a short row, a warp's 64 runs and a
    whole chunk of hub rows.  They weigh 0 beside the row's finite scores, forward and backward."""
    need_gpu()
    hg = lib()
    sp = hgsynth.spec("tiny-10k", n_user=2000, n_risk=10, num_rels=2, d=64)
    rng = np.random.default_rng(5)
    rels, offs, d = ((0, 1), (0, 0)), np.array([0, 2000, 2010], np.int64), 64
    # the rows' sources in run order, masked ones marked
    rows = [(range(96, 104), range(96, 100)), (range(0, 100), range(64, 100)), (range(200, 900), range(200, 712)),
            (range(1000, 1700), range(1512, 1700))]
    src = np.concatenate([np.array(s) for s, _ in rows]).astype(np.int32)
    dst = np.concatenate([np.full(len(s), 2000 + k) for k, (s, _) in enumerate(rows)]).astype(np.int32)
    w = SimpleNamespace(spec=sp, graph={"src": src, "dst": dst, "rel": np.zeros(src.size, np.int32),
                                        "type_offsets": offs, "rels": rels},
                        X=rng.standard_normal((2010, d)).astype(np.float32),
                        dH_top=rng.standard_normal((2010, d)).astype(np.float32))
    p = hgsynth.make_hgt_params(sp, 1)
    w.X[:, 0] = 0
    for _, masked in rows:
        w.X[list(masked), 0] = -1e30
    for k in ("W_K", "W_Q", "W_V", "W_att"):  # feature 0 reaches the keys alone, where it meets a query of 1e30
        p[k][..., 0, :] = 0
        p[k][..., :, 0] = 0
    p["W_K"][:, 0, 0] = p["W_att"][..., 0, 0] = 1
    p["b_K"][:, 0], p["b_Q"][:, 0] = 0, 1e30
    g = w.graph
    args = (g["src"], g["dst"], g["rel"], offs, rels, p, w.X)
    with np.errstate(under="ignore"):
        ref, _ = OH.hgt_forward(*args, 1, layernorm=False)
        dref, gref = OH.hgt_backward(*args, w.dH_top, 1, layernorm=False)
    out, dH, gr = run_gpu(hg, w, p, 1, False, w.dH_top)
    assert np.isfinite(out).all() and np.isfinite(dH).all()
    assert relerr(out[2000:], ref[2000:]) <= TOL["f32"]
    assert relerr(dH[:, 1:], dref[:, 1:]) <= TOL["f32"]
    for k in ("W_V", "W_msg", "W_agg", "b_V", "b_agg"):
        assert relerr(gr[k], gref[k]) <= TOL["f32"], k
    assert hg.hg_device_status() == 0


@pytest.mark.parametrize("into,dtype,d,heads", [(5, "f32", 64, 4), (5, "bf16", 128, 4), (8, "f32", 128, 8),
                                                (8, "bf16", 64, 2), (8, "bf16", 256, 4)])
def test_more_than_four_relations_into_a_type(into, dtype, d, heads):
    """Five to eight relations into the users (a claim holds four nodes, eight relation slots each): every subset of
    them occurs among the nodes, rows of one run, hub rows of one and of two chunks, live nodes not a multiple of 4."""
    need_gpu()
    hg = lib()
    nu, nr = 1201, 150
    rels = tuple((k % 2, 0) for k in range(into)) + ((0, 1),) * (into < 8)
    sp = hgsynth.spec("tiny-10k", n_user=nu, n_risk=nr, num_rels=len(rels), d=d, dtype=dtype)
    rng = np.random.default_rng(into * d)
    offs, sizes = np.array([0, nu, nu + nr], np.int64), (nu, nr)
    live = rng.permutation(nu)[: 4 * 220 + 3]
    src, dst, rel = [], [], []
    for r, (a, b) in enumerate(rels):
        if b == 0:  # target k has relation r when bit r of its place is set, and one to six edges then
            at = np.repeat(live[((np.arange(live.size) % (1 << into)) >> r) & 1 == 1], 3)
            at = np.concatenate([at, rng.choice(at, 2 * at.size)])
        else:
            at = offs[1] + rng.integers(0, nr, 400)
        src.append(offs[a] + rng.integers(0, sizes[a], at.size))
        dst.append(at)
        rel.append(np.full(at.size, r))
    hub = live[(1 << into) - 1]  # has every relation
    for r, runs in ((0, 700), (1, 120), (2, 97)):
        k = min(runs, sizes[rels[r][0]])
        src.append(offs[rels[r][0]] + rng.permutation(sizes[rels[r][0]])[:k])
        dst.append(np.full(k, hub))
        rel.append(np.full(k, r))
    g = {"src": np.concatenate(src).astype(np.int32), "dst": np.concatenate(dst).astype(np.int32),
         "rel": np.concatenate(rel).astype(np.int32), "type_offsets": offs, "rels": rels}
    assert np.unique(g["dst"][g["dst"] < nu]).size % 4
    st = hgsynth.bf16_round if dtype == "bf16" else (lambda x: x)
    w = SimpleNamespace(spec=sp, graph=g, X=st(rng.standard_normal((nu + nr, d)).astype(np.float32)),
                        dH_top=st(rng.standard_normal((nu + nr, d)).astype(np.float32)))
    p = hgsynth.make_hgt_params(sp, heads, bias_margin=BF16_RELU_MARGIN if dtype == "bf16" else None)
    out, dH, gr = run_gpu(hg, w, p, heads, True, w.dH_top)
    args = (g["src"], g["dst"], g["rel"], offs, rels, p, w.X)
    ref, _ = OH.hgt_forward(*args, heads, layernorm=True)
    dref, gref = OH.hgt_backward(*args, w.dH_top, heads, layernorm=True)
    assert relerr(out, ref) <= TOL[dtype], relerr(out, ref)
    assert relerr(dH, dref) <= TOL[dtype], relerr(dH, dref)
    for k in KEYS:
        assert relerr(gr[k], gref[k]) <= TOL[dtype], (k, relerr(gr[k], gref[k]))
    assert hg.hg_device_status() == 0


@pytest.mark.parametrize("dtype,d,many", [("f32", 64, False), ("bf16", 128, False), ("f32", 64, True), ("bf16", 64, True)])
def test_rows_around_the_hub_limits(dtype, d, many):
    """Rows and out-lists of 95 to 1025 runs, at the edges of a warp's share of a chunk and of a chunk; with many
    (above 16384 chunks) rows of up to 384 runs leave the chunks for a warp."""
    need_gpu()
    hg = lib()
    runs = [95, 96, 97, 124, 128, 129, 160, 161, 383, 384, 385, 511, 512, 513, 1024, 1025]
    fill = 17_000 if many else 0  # more rows of 97 runs
    nu, heads = 1100 + fill, 4
    rng = np.random.default_rng(d)
    src, dst = [], []
    for k, n in enumerate(runs):  # into risk k from n users, and from risk 20 + k into n users
        at = rng.permutation(1100)[:n]
        src += [at, np.full(n, nu + 20 + k)]
        dst += [np.full(n, nu + k), at]
    rel = np.concatenate([np.full(x.size, k % 2) for k, x in enumerate(src)])
    if many:  # hubs on both sides: the users from 1100 on have 97 in-edges each from 97 other users, and as many out-edges
        a = 1100 + np.repeat(np.arange(fill), 97)
        b = 1100 + (a - 1100 + 1 + np.tile(np.arange(97) * 3, fill)) % fill
        src.append(b), dst.append(a)
        rel = np.concatenate([rel, np.full(a.size, 2)])
    rels = ((0, 1), (1, 0), (0, 0))
    sp = hgsynth.spec("tiny-10k", n_user=nu, n_risk=40, num_rels=3, d=d, dtype=dtype)
    st = hgsynth.bf16_round if dtype == "bf16" else (lambda x: x)
    g = {"src": np.concatenate(src).astype(np.int32), "dst": np.concatenate(dst).astype(np.int32),
         "rel": rel.astype(np.int32), "type_offsets": np.array([0, nu, nu + 40], np.int64), "rels": rels}
    w = SimpleNamespace(spec=sp, graph=g, X=st(rng.standard_normal((nu + 40, d)).astype(np.float32)),
                        dH_top=st(rng.standard_normal((nu + 40, d)).astype(np.float32)))
    p = hgsynth.make_hgt_params(sp, heads, bias_margin=BF16_RELU_MARGIN)
    out, dH, gr = run_gpu(hg, w, p, heads, True, w.dH_top)
    args = (g["src"], g["dst"], g["rel"], g["type_offsets"], rels, p, w.X)
    ref, _ = OH.hgt_forward(*args, heads, layernorm=True)
    dref, gref = OH.hgt_backward(*args, w.dH_top, heads, layernorm=True)
    assert relerr(out, ref) <= TOL[dtype] and relerr(dH, dref) <= TOL[dtype]
    for k in KEYS:
        # every target has one relation, so b_K shifts all scores of a softmax alike: its gradient is zero
        scale = np.abs(gref["W_K" if k == "b_K" else k]).max()
        if k == "mu":  # <W_att, dW_att> / mu, a sum of cancelling terms
            scale = max(np.linalg.norm(p["W_att"][r]) * np.linalg.norm(gref["W_att"][r]) for r in range(3))
        assert np.abs(gr[k] - gref[k]).max() <= TOL[dtype] * scale, k
    assert hg.hg_device_status() == 0
