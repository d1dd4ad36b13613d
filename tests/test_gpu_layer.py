"""Layer forward / backward on the GPU against the oracle, element by element, on seeded inputs
that span several 64-row tiles, ragged tails and hub rows split into chunks."""
import numpy as np
import pytest
import torch

import hgsynth
import oracle
from tests.gpu_util import BF16_RELU_MARGIN, TOL, dev, grad_bufs, host, layer_params, lib, need_gpu, relerr, tdtype

pytestmark = pytest.mark.gpu

CASES = {
    # (workload, overrides): fp32 d=64 at full tiny size; bf16 d=128 / d=256 at reduced sizes of the
    # same recipes (power-law degrees with rows above the hub threshold, ragged type sizes)
    "tiny-f32-d64": ("tiny-10k", {}),
    "sub-bf16-d128": ("sub-1m", dict(n_user=27_001, n_risk=3_003, num_edges=600_000, n_overlap=4_000)),
    "tail-bf16-d256": ("tail-5m", dict(n_user=9_007, n_risk=1_001, num_edges=200_000, n_overlap=1_000, out_cap=4_000)),
    "tiny-bf16-d64": ("tiny-10k", dict(dtype="bf16")),
    "sub-f32-d128": ("sub-1m", dict(n_user=9_001, n_risk=1_003, num_edges=150_000, n_overlap=1_000, dtype="f32")),
}


def run_gpu_layer(hg, w, p, act, ln, dH_out):
    sp = w.spec
    g = w.graph
    td = tdtype(sp.dtype)
    G = hg.hg_build_csr(dev(g["src"]), dev(g["dst"]), dev(g["rel"]), g["type_offsets"], g["rels"])
    P = layer_params(hg, p, sp.dtype, act, ln)
    sb, kb = hg.hg_layer_workspace_size(G, P)
    saved = torch.empty(sb, dtype=torch.uint8, device="cuda")
    scratch = torch.empty(kb, dtype=torch.uint8, device="cuda")
    X = dev(w.X, td)
    out = torch.empty_like(X)
    hg.hg_layer_fwd(G, P, X, out, saved, scratch)
    dH_in = torch.empty_like(X)
    grads = grad_bufs(len(g["rels"]), 2, sp.d)
    hg.hg_layer_bwd(G, P, X, saved, dev(dH_out, td), dH_in, grads, scratch)
    torch.cuda.synchronize()
    return out, dH_in, grads


@pytest.mark.parametrize("case", list(CASES))
@pytest.mark.parametrize("act,ln", [("relu", True), ("relu", False), ("gelu_tanh", True)])
def test_layer_matches_oracle(case, act, ln):
    need_gpu()
    if act == "gelu_tanh" and case not in ("tiny-f32-d64", "sub-bf16-d128"):
        pytest.skip("activation variants covered on two shapes")
    hg = lib()
    name, ov = CASES[case]
    sp = hgsynth.spec(name, **ov)
    # bf16 ReLU: biases of +-8 (pre-activations have a spread of about 2) keep every pre-activation
    # clear of the kink, so that the kernel's decisions, taken on bf16-rounded intermediates, cannot
    # differ from the plain definition's (a single flipped decision moves a weight gradient, a sum
    # over all rows, by far more than the bf16 tolerance; see test_relu_near_zero_pre_activations)
    margin = BF16_RELU_MARGIN if (sp.dtype == "bf16" and act == "relu") else None
    w = hgsynth.make_workload(sp, random_affine=True, with_ids=False, bias_margin=margin)
    g = w.graph
    p = w.params[0]
    out, dH_in, grads = run_gpu_layer(hg, w, p, act, ln, w.dH_top)
    csr = oracle.build_csr(g["src"], g["dst"], g["rel"], g["type_offsets"], g["rels"])
    # the plain definition (Eq. 7, 10, 11 in fp64) for both storage types
    ref, _ = oracle.layer_forward(csr, g["type_offsets"], g["rels"], p, w.X, act, ln)
    tol = TOL[sp.dtype]
    assert relerr(host(out), ref) <= tol, ("H_out", relerr(host(out), ref))
    dref, gref = oracle.layer_backward(csr, g["type_offsets"], g["rels"], p, w.X, w.dH_top, act, ln)
    assert relerr(host(dH_in), dref) <= tol, ("dH_in", relerr(host(dH_in), dref))
    keys = ("W_rel", "W_agg", "b_agg") + (("ln_gamma", "ln_beta") if ln else ())
    for k in keys:
        e = relerr(host(grads[k]), gref[k])
        assert e <= tol, (k, e)
    assert hg.hg_device_status() == 0  # no bounded wait gave up


def test_layer_is_bitwise_repeatable():
    need_gpu()
    hg = lib()
    name, ov = CASES["sub-bf16-d128"]
    w = hgsynth.make_workload(hgsynth.spec(name, **ov), random_affine=True, with_ids=False)
    a = run_gpu_layer(hg, w, w.params[0], "relu", True, w.dH_top)
    b = run_gpu_layer(hg, w, w.params[0], "relu", True, w.dH_top)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    for k in a[2]:
        assert torch.equal(a[2][k], b[2][k]), k


def test_layer_without_edges_and_without_dH_in():
    need_gpu()
    hg = lib()
    sp = hgsynth.spec("tiny-10k", n_user=700, n_risk=90, num_edges=0, n_overlap=50)
    w = hgsynth.make_workload(sp, random_affine=True, with_ids=False)
    g = w.graph
    p = w.params[0]
    G = hg.hg_build_csr(dev(g["src"]), dev(g["dst"]), dev(g["rel"]), g["type_offsets"], g["rels"])
    P = layer_params(hg, p, sp.dtype)
    sb, kb = hg.hg_layer_workspace_size(G, P)
    saved = torch.empty(sb, dtype=torch.uint8, device="cuda")
    scratch = torch.empty(kb, dtype=torch.uint8, device="cuda")
    X = dev(w.X, torch.float32)
    out = torch.empty_like(X)
    hg.hg_layer_fwd(G, P, X, out, saved, scratch)
    grads = grad_bufs(len(g["rels"]), 2, sp.d)
    hg.hg_layer_bwd(G, P, X, saved, dev(w.dH_top, torch.float32), None, grads, scratch)
    csr = oracle.build_csr(g["src"], g["dst"], g["rel"], g["type_offsets"], g["rels"])
    ref, _ = oracle.layer_forward(csr, g["type_offsets"], g["rels"], p, w.X)
    assert relerr(host(out), ref) <= 1e-5
    _, gref = oracle.layer_backward(csr, g["type_offsets"], g["rels"], p, w.X, w.dH_top)
    for k in gref:
        assert relerr(host(grads[k]), gref[k]) <= 1e-5 or np.abs(gref[k]).max() == 0, k
        if np.abs(gref[k]).max() == 0:
            assert host(grads[k]).max() == 0 and host(grads[k]).min() == 0, k


def test_relu_near_zero_pre_activations_bf16():
    """bf16, ReLU, biases near zero: many pre-activations lie within a rounding of zero, where the
    mask of either side is a valid outcome of bf16 storage.  This is the one comparison with the
    oracle's bf16-storage mode (M_r and U rounded where the kernel stores them, so both sides decide
    on the same values).  Row outputs (H_out, dH_in) and the LayerNorm gradients are compared at the
    bf16 tolerance; the weight gradients, sums over all rows in which a few such decisions may
    differ, are compared in the Frobenius norm."""
    need_gpu()
    hg = lib()
    name, ov = CASES["sub-bf16-d128"]
    sp = hgsynth.spec(name, **ov)
    w = hgsynth.make_workload(sp, random_affine=True, with_ids=False)
    g = w.graph
    p = w.params[0]
    out, dH_in, grads = run_gpu_layer(hg, w, p, "relu", True, w.dH_top)
    csr = oracle.build_csr(g["src"], g["dst"], g["rel"], g["type_offsets"], g["rels"])
    ref, _ = oracle.layer_forward(csr, g["type_offsets"], g["rels"], p, w.X, "relu", True, store="bf16")
    dref, gref = oracle.layer_backward(csr, g["type_offsets"], g["rels"], p, w.X, w.dH_top, "relu", True, store="bf16")
    assert relerr(host(out), ref) <= 2e-2
    assert relerr(host(dH_in), dref) <= 2e-2
    for k in ("ln_gamma", "ln_beta"):
        assert relerr(host(grads[k]), gref[k]) <= 2e-2, k
    for k in ("W_rel", "W_agg", "b_agg"):
        x, y = host(grads[k]), gref[k]
        assert np.linalg.norm(x - y) / np.linalg.norm(y) <= 2e-2, k


@pytest.mark.parametrize("d,ln,idle", [(128, True, 0), (128, True, 127), (128, False, 128), (128, True, 129),
                                       (128, True, 400), (64, True, 128), (64, False, 400), (256, True, 129)])
def test_nodes_without_in_edges_bf16(d, ln, idle):
    """`idle` of 400 users and every risk node without in-edges: whole 128-row tiles of them leave the projection."""
    need_gpu()
    hg = lib()
    sp = hgsynth.spec("tiny-10k", n_user=400, n_risk=100, num_edges=6_000, n_overlap=10, dtype="bf16", d=d)
    w = hgsynth.make_workload(sp, random_affine=True, with_ids=False, bias_margin=BF16_RELU_MARGIN)
    g, p = w.graph, w.params[0]
    keep = np.flatnonzero(g["rel"] == 0) if idle < 400 else np.zeros(0, np.int64)  # relation 0: user -> user
    for k in ("src", "dst", "rel"):
        g[k] = np.ascontiguousarray(g[k][keep])
    targets = np.random.default_rng(0).permutation(400)[: 400 - idle]
    if keep.size:
        g["dst"] = targets[np.arange(keep.size) % targets.size].astype(g["dst"].dtype)
    out, dH_in, grads = run_gpu_layer(hg, w, p, "relu", ln, w.dH_top)
    csr = oracle.build_csr(g["src"], g["dst"], g["rel"], g["type_offsets"], g["rels"])
    ref, _ = oracle.layer_forward(csr, g["type_offsets"], g["rels"], p, w.X, "relu", ln)
    dref, gref = oracle.layer_backward(csr, g["type_offsets"], g["rels"], p, w.X, w.dH_top, "relu", ln)
    assert relerr(host(out), ref) <= TOL["bf16"] and relerr(host(dH_in), dref) <= TOL["bf16"]
    for k in ("W_rel", "W_agg", "b_agg") + (("ln_gamma", "ln_beta") if ln else ()):
        assert np.abs(host(grads[k]) - gref[k]).max() <= TOL["bf16"] * np.abs(gref[k]).max(), k
    assert hg.hg_device_status() == 0


@pytest.mark.parametrize("kind", ["mean", "attention"])
@pytest.mark.parametrize("dt", ["f32", "bf16"])
def test_scratch_for_hub_partials_follows_the_rows(kind, dt):
    """400 rows and a million edges: room for a chunk per 512 runs and one more per row, once, in both layers."""
    need_gpu()
    hg = lib()
    n, d, heads, E = 400, 64, 4, 1_000_000
    offs, rels = np.array([0, n, n], np.int64), ((0, 0),)
    sp = hgsynth.spec("tiny-10k", n_user=n, n_risk=0, num_rels=1, d=d, dtype=dt)
    size = {}
    for edges in (1, E):
        e = dev(np.zeros(edges, np.int32))
        G = hg.hg_build_csr(e, e, e, offs, rels)
        if kind == "mean":
            P = layer_params(hg, hgsynth.make_layer_params(sp, 0), dt)
            size[edges] = hg.hg_layer_workspace_size(G, P)[1]
        else:
            p = hgsynth.make_hgt_params(sp, heads)
            P = hg.HgtParams({k: dev(v, torch.float32 if k == "mu" else tdtype(dt)) for k, v in p.items()}, heads)
            size[edges] = hg.hg_hgt_workspace_size(G, P)[1]
    partial = d if kind == "mean" else max(2 * heads + d, 2 * d)
    assert size[E] - size[1] <= (E // 512 + n) * partial * 4 + 256
