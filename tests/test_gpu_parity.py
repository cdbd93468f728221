"""GPU parity: every stage of the CUDA path against the CPU oracle, through the C ABI.

Stage tests feed each GPU stage the oracle's output of the previous one ("teacher forcing"),
so integer stages are compared bit for bit.  End-to-end tests run the fused call and account
for near-tie swaps.  All inputs come from the seeded generator; the oracle reads the bytes the
GPU read.
"""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2605_26678_b200 import nkv
from paper_2605_26678_b200 import workloads as wl
from tests import parity as pr

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _cache(N, d, dtype, H=2, layers=1, seed=11, seg=(32, 96)):
    cfg = wl.tiny_config(kv_heads=H, head_dim=d, seq_len=N, dtype=dtype, layers=layers, base_seed=seed,
                         seg_lo=seg[0], seg_hi=seg[1])
    K, V = wl.make_cache(cfg)
    return K.to(DEV), V.to(DEV)


SHAPES = [(1, 64, "fp32"), (3, 64, "bf16"), (63, 128, "bf16"), (64, 64, "fp32"), (65, 128, "fp32"),
          (200, 64, "bf16"), (257, 128, "bf16"), (1000, 128, "fp32"), (4133, 64, "bf16"), (6000, 128, "bf16"),
          (300, 64, "fp16"), (4133, 128, "fp16")]


@pytest.mark.parametrize("N,d,dtype", SHAPES)
def test_anchors_match_oracle(N, d, dtype):
    K, _ = _cache(N, d, dtype)
    mu_s, mu_e, inv_norm, mu_c = nkv.nkv_anchors(K, want_mu_c=(N <= 1000))
    torch.cuda.synchronize()
    for g in range(K.shape[0]):
        for h in range(K.shape[1]):
            ref = oracle.score_head(K[g, h].cpu(), want_mu_c=(N <= 1000))
            pr.assert_close(inv_norm[g, h].cpu().numpy(), ref.inv_norm, "inv_norm", 1e-5)
            pr.assert_close(mu_s[g, h].cpu().numpy(), ref.mu_s, "mu_s", 1e-5)
            pr.assert_close(mu_e[g, h].cpu().numpy(), ref.mu_e, "mu_e", 1e-5)
            if mu_c is not None:
                pr.assert_close(mu_c[g, h].cpu().numpy(), ref.mu_c, "mu_c", 1e-5)


@pytest.mark.parametrize("N,d,dtype", SHAPES)
def test_scores_match_oracle(N, d, dtype):
    K, _ = _cache(N, d, dtype)
    mu_s, mu_e, inv_norm, _ = nkv.nkv_anchors(K)
    a_star, a_raw, stats = nkv.nkv_score(K, mu_s, mu_e, inv_norm, want_raw=True, want_stats=True)
    torch.cuda.synchronize()
    for h in range(K.shape[1]):
        ref = oracle.score_head(K[0, h].cpu())
        pr.assert_close(a_raw[0, h].cpu().numpy(), ref.a_raw, "a_raw")
        st = stats[0, h].cpu().numpy()
        if N >= 8:   # with a handful of tokens the min-max range can be rounding noise in both precisions
            pr.assert_close(st[0:3], ref.lo, "lo")
            pr.assert_close(st[3:6], ref.hi, "hi")
            pr.assert_close(st[6:9], ref.delta, "delta")
            pr.assert_close(st[9:12], ref.w, "w")
            pr.assert_close(st[12:15], [ref.s_min, ref.s_max, ref.s_mean], "surprise stats")
            pr.assert_close(a_star[0, h].cpu().numpy(), ref.a_star, "a_star")
        assert st[15] == ref.m
        assert torch.isinf(a_star[0, h, :min(4, N)]).all()


KEY_SCAN_CASES = [("fma", 1, 64, "fp32"), ("fma", 63, 128, "bf16"), ("fma", 257, 128, "bf16"), ("fma", 1000, 128, "fp32"),
                  ("fma", 4133, 64, "bf16"), ("fma", 6000, 128, "bf16"), ("tensor", 100, 128, "bf16"),
                  ("tensor", 257, 128, "bf16"), ("tensor", 2500, 128, "bf16"), ("tensor", 4352, 128, "bf16"),
                  ("tensor", 8200, 128, "bf16"), ("tensor", 4133, 64, "bf16"), ("auto", 3000, 128, "bf16"),
                  ("auto", 2500, 128, "fp16"), ("tensor", 777, 64, "fp16")]


@pytest.mark.parametrize("mode,N,d,dtype", KEY_SCAN_CASES)
def test_key_scan_intermediates_match_oracle(mode, N, d, dtype):
    """The kernels nkv_compress times, stage by stage: 1/||k||, the anchors, the three raw anomalies and their
    per-head extremes straight out of the key scan, for the FMA and the tensor-core form."""
    K, _ = _cache(N, d, dtype, H=3)
    p = nkv.nkv_default_params()
    ws = nkv.alloc_workspace(K, p)
    nkv.nkv_set_key_passes(mode)
    try:
        inv_norm, mu_s, mu_e, a_raw, minmax = nkv.nkv_key_scan(K, p, ws=ws)
    finally:
        nkv.nkv_set_key_passes("auto")
    assert nkv.nkv_last_device_status(ws) == nkv.NKV_OK
    for h in range(K.shape[1]):
        ref = oracle.score_head(K[0, h].cpu())
        pr.assert_close(inv_norm[0, h].cpu().numpy(), ref.inv_norm, "inv_norm", 1e-5)
        pr.assert_close(mu_s[0, h].cpu().numpy(), ref.mu_s, "mu_s", 1e-5)
        pr.assert_close(mu_e[0, h].cpu().numpy(), ref.mu_e, "mu_e", 1e-5)
        pr.assert_close(a_raw[0, h].cpu().numpy(), ref.a_raw, "a_raw", 1e-5)
        mm = minmax[0, h].cpu().numpy()
        pr.assert_close(mm[0::2], ref.lo, "lo", 1e-5)
        pr.assert_close(mm[1::2], ref.hi, "hi", 1e-5)


@pytest.mark.parametrize("prior,gate", [((1.0, 0.0, 0.0), nkv.NKV_GATE_AVERAGE), ((0.5, 0.5, 0.0), nkv.NKV_GATE_AVERAGE),
                                        ((0.5, 0.5, 0.0), nkv.NKV_GATE_SURPRISE), ((0.0, 0.0, 1.0), nkv.NKV_GATE_MAX)])
def test_ablation_priors_switch_scales_off(prior, gate):
    """Single-anchor scoring (the "w/o continuum" row of the ablation table) and scoring without the current
    memory (the components table): a prior of zero removes a scale from the blend."""
    K, V = _cache(1500, 128, "bf16", H=2)
    p = nkv.nkv_default_params()
    p.gate_mode = gate
    for k in range(3):
        p.prior[k] = prior[k]
    res = nkv.nkv_compress(K, V, 0.75, p, want_a_star=True)
    torch.cuda.synchronize()
    for h in range(K.shape[1]):
        ref = oracle.score_head(K[0, h].cpu(), pr.oracle_params(p))
        assert [w == 0.0 for w in ref.w] == [x == 0.0 for x in prior]
        pr.assert_close(res.a_star[0, h].cpu().numpy(), ref.a_star, "a_star")
    if prior == (1.0, 0.0, 0.0):   # key distinctiveness: min-max of -cos(k_hat, mean k_hat)
        a = res.a_star[0, 0, 4:].cpu().numpy()
        ref = oracle.score_head(K[0, 0].cpu())
        want = (ref.a_raw[0] - ref.lo[0]) / (ref.hi[0] - ref.lo[0])
        pr.assert_close(a, want[4:], "single-anchor score")


@pytest.mark.parametrize("gate,window,n_sink,prior", [
    (nkv.NKV_GATE_AVERAGE, 64, 4, (0.4, 0.4, 0.2)), (nkv.NKV_GATE_MAX, 64, 0, (0.4, 0.4, 0.2)),
    (nkv.NKV_GATE_SURPRISE, 2, 4, (0.2, 0.3, 0.5)), (nkv.NKV_GATE_SURPRISE, 17, 8, (0.4, 0.4, 0.2)),
    (nkv.NKV_GATE_SURPRISE, 40, 16, (0.6, 0.3, 0.1))])
def test_score_parameter_switches(gate, window, n_sink, prior):
    K, _ = _cache(777, 128, "bf16")
    p = nkv.nkv_default_params()
    p.gate_mode, p.window, p.n_sink = gate, window, n_sink
    p.block_div, p.block_min, p.block_max = 64, 64, 128
    p.beta, p.tau, p.kappa = 2.0, 0.3, 6.0
    for k in range(3):
        p.prior[k] = prior[k]
    mu_s, mu_e, inv_norm, _ = nkv.nkv_anchors(K, p)
    a_star, a_raw, _ = nkv.nkv_score(K, mu_s, mu_e, inv_norm, p, want_raw=True)
    torch.cuda.synchronize()
    for h in range(K.shape[1]):
        ref = oracle.score_head(K[0, h].cpu(), pr.oracle_params(p))
        pr.assert_close(a_raw[0, h].cpu().numpy(), ref.a_raw, "a_raw")
        pr.assert_close(a_star[0, h].cpu().numpy(), ref.a_star, "a_star")


def _random_scores(G, H, N, seed, ties):
    rng = np.random.default_rng(seed)
    s = rng.random((G, H, N)).astype(np.float32) ** 3
    s *= rng.uniform(0.05, 1.0, size=(G, H, 1)).astype(np.float32)
    if ties == "many":
        s = np.round(s * 16) / 16
    elif ties == "all":
        s[:] = 0.25
    elif ties == "dense":          # bulk packed into a sliver of [0,1], like real scores
        s = (0.05 + 0.001 * s).astype(np.float32)
    s[:, :, :4] = np.inf
    return s


@pytest.mark.parametrize("G,H,N,r,ties", [
    (1, 1, 10, 0.5, "none"), (2, 3, 100, 0.75, "none"), (1, 8, 1000, 0.75, "many"), (2, 4, 5000, 0.95, "dense"),
    (1, 8, 3000, 0.5, "all"), (1, 2, 4097, 0.0, "none"), (3, 8, 2048, 0.9, "dense"), (1, 5, 40, 0.95, "none"),
    # large enough for the parallel form of the group competition; "dense" and "all" overflow its candidate list
    (2, 8, 20000, 0.75, "none"), (2, 8, 12000, 0.5, "many"), (1, 8, 16384, 0.95, "dense"), (1, 8, 9000, 0.5, "all"),
    (3, 5, 14001, 0.9, "none")])
def test_budget_and_select_bit_exact_on_oracle_scores(G, H, N, r, ties):
    s = _random_scores(G, H, N, seed=N + H, ties=ties)
    a_star = torch.from_numpy(s).to(DEV)
    budgets = nkv.nkv_budget(a_star, r)
    k = nkv.nkv_keep_per_head(N, r)
    idx, offs, ranks = nkv.nkv_select(a_star, budgets, H * k, want_ranks=(N <= 5000))
    torch.cuda.synchronize()
    for g in range(G):
        ref = oracle.budget_select(s[g], r, want_ranks=True)
        assert np.array_equal(budgets[g].cpu().numpy(), ref.budgets)
        assert np.array_equal(offs[g].cpu().numpy(), ref.offsets)
        assert np.array_equal(idx[g].cpu().numpy(), ref.idx)
        if ranks is not None:
            assert np.array_equal(ranks[g].cpu().numpy(), ref.ranks)


def test_safeguard_one_gives_uniform_budgets():
    s = _random_scores(2, 4, 600, seed=3, ties="none")
    p = nkv.nkv_default_params()
    p.safeguard = 1.0
    budgets = nkv.nkv_budget(torch.from_numpy(s).to(DEV), 0.75, p)
    assert budgets.cpu().tolist() == [[150] * 4] * 2


@pytest.mark.parametrize("d,dv,dtype,mode", [(128, 128, "bf16", "out"), (64, 64, "fp32", "out"),
                                             (128, 128, "fp32", "in"), (64, 64, "bf16", "in"),
                                             (128, 64, "bf16", "out"), (64, 128, "fp32", "out"),
                                             (128, 64, "bf16", "in"), (128, 128, "fp16", "out")])
def test_compaction_copies_rows_verbatim(d, dv, dtype, mode):
    K, V = _cache(900, d, dtype, H=3, layers=2)
    if dv != d:   # values of another width (the paper's V in R^{N x d_v}): same rows, other row length
        V = _cache(900, dv, dtype, H=3, layers=2, seed=12)[1]
    s = _random_scores(2, 3, 900, seed=5, ties="none")
    sel = [oracle.budget_select(s[g], 0.6) for g in range(2)]
    idx = torch.from_numpy(np.stack([x.idx for x in sel])).to(DEV)
    offs = torch.from_numpy(np.stack([x.offsets for x in sel])).to(DEV)
    Kr, Vr = pr.raw_rows(K), pr.raw_rows(V)
    if mode == "out":
        K_out, V_out = nkv.nkv_compact(K, V, idx, offs)
        torch.cuda.synchronize()
        for g in range(2):
            assert np.array_equal(pr.raw_rows(K_out[g]), oracle.compact(K[g].cpu(), sel[g].idx, sel[g].offsets))
            assert np.array_equal(pr.raw_rows(V_out[g]), oracle.compact(V[g].cpu(), sel[g].idx, sel[g].offsets))
    else:
        Kc, Vc = K.clone(), V.clone()
        nkv.nkv_compact(Kc, Vc, idx, offs, mode=nkv.NKV_IN_PLACE)
        torch.cuda.synchronize()
        Kg, Vg = pr.raw_rows(Kc), pr.raw_rows(Vc)
        for g in range(2):
            for h in range(3):
                rows = sel[g].idx[sel[g].offsets[h]:sel[g].offsets[h + 1]]
                assert np.array_equal(Kg[g, h, :len(rows)], Kr[g, h][rows])
                assert np.array_equal(Vg[g, h, :len(rows)], Vr[g, h][rows])


@pytest.mark.parametrize("N,d,dtype,H,layers,r", [
    (5, 64, "fp32", 2, 1, 0.5), (300, 64, "bf16", 4, 2, 0.75), (1000, 128, "fp32", 8, 1, 0.5),
    (2500, 128, "bf16", 8, 2, 0.95), (4133, 64, "bf16", 3, 1, 0.0), (777, 128, "bf16", 1, 3, 0.9),
    (3000, 128, "fp16", 4, 2, 0.85), (900, 64, "fp16", 2, 1, 0.25)])
def test_fused_compress_end_to_end(N, d, dtype, H, layers, r):
    K, V = _cache(N, d, dtype, H=H, layers=layers)
    p = nkv.nkv_default_params()
    ws = nkv.alloc_workspace(K, p)
    res = nkv.nkv_compress(K, V, r, p, ws=ws, want_a_star=True)
    assert nkv.nkv_last_device_status(ws) == nkv.NKV_OK
    rep = pr.SwapReport()
    for g in range(K.shape[0]):
        pr.check_group_against_oracle(K, V, res, g, r, p, rep)
    assert rep.swapped_tokens <= max(2, rep.heads)   # near-tie swaps are rare at fp32 accuracy


@pytest.mark.parametrize("N,H,layers,r", [
    (100, 2, 1, 0.5), (777, 1, 3, 0.9), (2500, 8, 2, 0.95), (4096, 4, 1, 0.75), (8200, 3, 1, 0.75),
    (4352, 2, 1, 0.75), (6144, 2, 1, 0.5)])   # the last two: blocks of 136 and 192 keys straddle the 128-key tiles
@pytest.mark.parametrize("mode,d", [("tensor", 128), ("fma", 128), ("tensor", 64)])
def test_key_pass_kernels_end_to_end(N, H, layers, r, mode, d):
    """Both key passes on the tensor cores (tcgen05: band sums of the keys' Gram matrix, dots with the
    split anchors) and both as FMA kernels, each against the oracle.  With d = 64 only the second pass
    has a tensor-core form."""
    K, V = _cache(N, d, "bf16", H=H, layers=layers)
    p = nkv.nkv_default_params()
    ws = nkv.alloc_workspace(K, p)
    before = nkv.nkv_launch_count()
    nkv.nkv_set_key_passes(mode)
    try:
        res = nkv.nkv_compress(K, V, r, p, ws=ws, want_a_star=True)
    finally:
        nkv.nkv_set_key_passes("auto")
    assert nkv.nkv_last_device_status(ws) == nkv.NKV_OK
    assert nkv.nkv_launch_count() > before
    rep = pr.SwapReport()
    for g in range(K.shape[0]):
        pr.check_group_against_oracle(K, V, res, g, r, p, rep)
    assert rep.swapped_tokens <= max(2, rep.heads)


@pytest.mark.parametrize("N,d,dtype,H,layers,r", [(600, 128, "bf16", 2, 9, 0.75), (333, 64, "fp32", 3, 10, 0.5)])
def test_many_groups_and_repeated_calls(N, d, dtype, H, layers, r):
    """Nine and ten layer groups in one call: every group matches the oracle, and two calls in a row on
    the same buffers and workspace give identical outputs (nothing is left over from the first)."""
    K, V = _cache(N, d, dtype, H=H, layers=layers)
    p = nkv.nkv_default_params()
    ws = nkv.alloc_workspace(K, p)
    res = nkv.nkv_compress(K, V, r, p, ws=ws, want_a_star=True)
    torch.cuda.synchronize()
    assert nkv.nkv_last_device_status(ws) == nkv.NKV_OK
    first = (res.idx.clone(), res.k_out.clone(), res.v_out.clone(), res.budgets.clone())
    rep = pr.SwapReport()
    for g in range(K.shape[0]):
        pr.check_group_against_oracle(K, V, res, g, r, p, rep)
    assert rep.swapped_tokens <= max(2, rep.heads)
    res = nkv.nkv_compress(K, V, r, p, out=res, ws=ws)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(first, (res.idx, res.k_out, res.v_out, res.budgets)))


def test_identical_keys_take_the_tie_path():
    """All keys equal: every score is 0 and every selection is decided by position alone."""
    K = torch.ones((1, 2, 3000, 64), dtype=torch.bfloat16, device=DEV)
    V = torch.randn((1, 2, 3000, 64), device=DEV).to(torch.bfloat16)
    ws = nkv.alloc_workspace(K)
    res = nkv.nkv_compress(K, V, 0.75, ws=ws, want_a_star=True)
    assert nkv.nkv_last_device_status(ws) == nkv.NKV_OK
    a = res.a_star.cpu().numpy()
    assert np.isinf(a[0, :, :4]).all() and (a[0, :, 4:] == 0).all()
    ref = oracle.budget_select(a[0], 0.75)
    assert np.array_equal(res.budgets[0].cpu().numpy(), ref.budgets)
    assert np.array_equal(res.idx[0].cpu().numpy(), ref.idx)


def test_strided_heads_outermost_layout():
    """A [H, G, N, d] allocation viewed as [G, H, N, d]: strides, not copies."""
    K, V = _cache(600, 128, "bf16", H=3, layers=2)
    Kt = K.permute(1, 0, 2, 3).contiguous().permute(1, 0, 2, 3)
    Vt = V.permute(1, 0, 2, 3).contiguous().permute(1, 0, 2, 3)
    assert not Kt.is_contiguous()
    a = nkv.nkv_compress(K, V, 0.75, want_a_star=True)
    b = nkv.nkv_compress(Kt, Vt, 0.75, want_a_star=True)
    torch.cuda.synchronize()
    assert torch.equal(a.idx, b.idx) and torch.equal(a.k_out, b.k_out) and torch.equal(a.v_out, b.v_out)
    assert torch.equal(a.a_star, b.a_star)


def test_argument_errors_are_reported_not_thrown():
    K, V = _cache(100, 64, "fp32")
    with pytest.raises(nkv.NkvError) as e:
        nkv.nkv_compress(K, V, 1.0)
    assert e.value.status == nkv.NKV_ERR_INVALID_ARG
    with pytest.raises(nkv.NkvError) as e:
        nkv.nkv_compress(K, V, 0.999)      # k = 0
    assert e.value.status == nkv.NKV_ERR_INVALID_ARG
    with pytest.raises(nkv.NkvError) as e:
        nkv.nkv_compress(K[..., :48].contiguous(), V[..., :48].contiguous(), 0.5)
    assert e.value.status == nkv.NKV_ERR_UNSUPPORTED
    for bad_window in (65, 1, 0):
        p = nkv.nkv_default_params()
        p.window = bad_window
        with pytest.raises(nkv.NkvError) as e:
            nkv.nkv_compress(K, V, 0.5, p)
        assert e.value.status == nkv.NKV_ERR_UNSUPPORTED
    p = nkv.nkv_default_params()
    p.prior[0] = p.prior[1] = p.prior[2] = 0.0
    with pytest.raises(nkv.NkvError) as e:
        nkv.nkv_compress(K, V, 0.5, p)
    assert e.value.status == nkv.NKV_ERR_INVALID_ARG
    with pytest.raises(nkv.NkvError) as e:
        nkv.nkv_compress(K, V, 0.5, ws=torch.empty(1024, dtype=torch.uint8, device=DEV))
    assert e.value.status == nkv.NKV_ERR_WORKSPACE
    with pytest.raises(nkv.NkvError) as e:
        nkv.nkv_compress(K.double(), V.double(), 0.5)
    assert e.value.status == nkv.NKV_ERR_UNSUPPORTED


def test_host_buffer_entry_point_matches_device_entry_point():
    K, V = _cache(1500, 128, "bf16", H=4, layers=5)
    dev = nkv.nkv_compress(K, V, 0.75)
    torch.cuda.synchronize()
    Kh, Vh = K.cpu().pin_memory(), V.cpu().pin_memory()
    G, H, N, d = K.shape
    k = nkv.nkv_keep_per_head(N, 0.75)
    out = nkv.Compressed(torch.empty((G, H * k, d), dtype=K.dtype).pin_memory(),
                         torch.empty((G, H * k, d), dtype=K.dtype).pin_memory(),
                         torch.empty((G, H * k), dtype=torch.int32).pin_memory(),
                         torch.empty((G, H + 1), dtype=torch.int32).pin_memory(),
                         torch.empty((G, H), dtype=torch.int32).pin_memory(), None)
    nbytes = nkv.nkv_host_staging_bytes(H, N, d, nkv.NKV_BF16, 0.75, 2)
    staging = torch.empty(nbytes, dtype=torch.uint8, device=DEV)
    nkv.nkv_compress_host(Kh, Vh, 0.75, out, staging, 2)
    assert torch.equal(out.idx, dev.idx.cpu()) and torch.equal(out.budgets, dev.budgets.cpu())
    assert torch.equal(out.head_offsets, dev.head_offsets.cpu())
    assert torch.equal(out.k_out, dev.k_out.cpu()) and torch.equal(out.v_out, dev.v_out.cpu())


def test_too_many_heads_is_an_argument_error():
    """More than 65535 heads in one call is refused before anything is launched."""
    K = torch.zeros((8200, 8, 1, 64), dtype=torch.bfloat16, device=DEV)
    before = nkv.nkv_launch_count()
    with pytest.raises(nkv.NkvError) as e:
        nkv.nkv_compress(K, K, 0.0)
    assert e.value.status == nkv.NKV_ERR_UNSUPPORTED
    assert nkv.nkv_launch_count() == before


def test_host_entry_point_reports_a_device_status_of_any_chunk():
    """A device-side status raised while any chunk runs comes back from nkv_compress_host: the status words
    of every chunk are copied out before the chunk's slot is reused.  The status is planted by the library's
    test hook, nothing on the device misbehaves."""
    K, V = _cache(600, 64, "bf16", H=2, layers=6)
    Kh, Vh = K.cpu().pin_memory(), V.cpu().pin_memory()
    G, H, N, d = K.shape
    k = nkv.nkv_keep_per_head(N, 0.5)
    out = nkv.Compressed(torch.empty((G, H * k, d), dtype=K.dtype).pin_memory(),
                         torch.empty((G, H * k, d), dtype=K.dtype).pin_memory(),
                         torch.empty((G, H * k), dtype=torch.int32).pin_memory(),
                         torch.empty((G, H + 1), dtype=torch.int32).pin_memory(),
                         torch.empty((G, H), dtype=torch.int32).pin_memory(), None)
    staging = torch.empty(nkv.nkv_host_staging_bytes(H, N, d, nkv.NKV_BF16, 0.5, 2), dtype=torch.uint8, device=DEV)
    nkv.nkv_compress_host(Kh, Vh, 0.5, out, staging, 2)           # three chunks, all fine
    for chunk, code in ((0, nkv.NKV_ERR_TIMEOUT), (1, nkv.NKV_ERR_DEVICE_CHECK), (2, nkv.NKV_ERR_TIMEOUT)):
        nkv.nkv_debug_set("inject_host_status", chunk * 16 + code)
        try:
            with pytest.raises(nkv.NkvError) as e:
                nkv.nkv_compress_host(Kh, Vh, 0.5, out, staging, 2)
            assert e.value.status == code
        finally:
            nkv.nkv_debug_set("inject_host_status", 0)
    nkv.nkv_compress_host(Kh, Vh, 0.5, out, staging, 2)           # and fine again


@pytest.mark.gpu
def test_a_wait_that_runs_out_is_reported_and_leaves_the_device_usable():
    """The hand-overs of the tensor-core key passes are bounded mbarrier waits.  The probe runs that same wait on a
    barrier nothing arrives at: it must end by itself, the status words must say NKV_ERR_TIMEOUT with the probe's
    detail code, and the next ordinary call on the same workspace must be clean."""
    cfg = wl.CONFIGS["cfg1_single_layer_fp32_4k"]
    K, V = wl.make_cache(cfg, "cuda:0")
    p = nkv.nkv_default_params()
    ws = nkv.alloc_workspace(K, p)
    nkv.nkv_debug_wait_probe(2000, ws)
    assert nkv.nkv_last_device_status(ws) == nkv.NKV_ERR_TIMEOUT
    words = ws[:16].view(torch.int32).cpu().tolist()
    assert words[0] == nkv.NKV_ERR_TIMEOUT and 799 in words[:4]
    with pytest.raises(nkv.NkvError):
        nkv.nkv_debug_wait_probe(0, ws)
    out = nkv.nkv_compress(K, V, 0.75, p, ws=ws)
    assert nkv.nkv_last_device_status(ws) == nkv.NKV_OK
    assert int(out.budgets.sum()) == K.shape[1] * nkv.nkv_keep_per_head(K.shape[2], 0.75)


@pytest.mark.gpu
@pytest.mark.parametrize("r", [0.5, 0.75, 0.95])
def test_budget_thresholds_bracket_the_budgets(r):
    """nkv_budget's optional thresholds: per head, the tokens scoring above the threshold fit into the budget and the
    tokens scoring at least the threshold fill it (Section 2.6: the threshold is the score of the last slot taken)."""
    g = torch.Generator(device="cpu").manual_seed(11)
    G, H, N = 3, 8, 5000
    a = torch.rand((G, H, N), generator=g, dtype=torch.float32)
    a[:, :, ::7] = a[:, :, 1::7][:, :, : a[:, :, ::7].shape[2]]   # plant exact ties
    a[:, :, :4] = float("inf")
    a_dev = a.cuda()
    budgets, thr = nkv.nkv_budget(a_dev, r, want_thresholds=True)
    assert torch.equal(budgets.cpu(), nkv.nkv_budget(a_dev, r).cpu())
    above = (a_dev > thr[:, :, None]).sum(dim=2)
    at_least = (a_dev >= thr[:, :, None]).sum(dim=2)
    assert bool((above <= budgets).all()) and bool((budgets <= at_least).all())
    assert int(budgets.sum()) == G * H * nkv.nkv_keep_per_head(N, r)


@pytest.mark.gpu
@pytest.mark.parametrize("seed", [7, 23])
def test_random_shapes_end_to_end(seed):
    """Twenty seeded random calls per seed (N from 65 to 12000 with tile-aligned and ragged lengths, d, storage, heads,
    layers, ratio and key-pass form drawn at random), each compared with the oracle group by group."""
    import random
    rng = random.Random(seed)
    p = nkv.nkv_default_params()
    swaps = heads = 0
    for case in range(20):
        d = rng.choice([64, 128, 128])
        dtype = rng.choice(["bf16", "bf16", "fp16", "fp32"])
        N = rng.choice([rng.randint(65, 700), rng.randint(700, 5000), rng.randint(5000, 12000), 128 * rng.randint(1, 40),
                        256 * rng.randint(1, 20) + rng.choice([0, 1, 127])])
        H, layers = rng.randint(1, 8), rng.randint(1, 3)
        r = rng.choice([0.25, 0.5, 0.75, 0.85, 0.95])
        mode = rng.choice(["auto", "tensor", "tensor", "fma"])
        if nkv.nkv_keep_per_head(N, r) < 1:
            continue
        K, V = _cache(N, d, dtype, H=H, layers=layers, seed=100 * seed + case, seg=(32, rng.choice([96, 400, 2000])))
        ws = nkv.alloc_workspace(K, p)
        nkv.nkv_set_key_passes(mode)
        try:
            res = nkv.nkv_compress(K, V, r, p, ws=ws, want_a_star=True)
        finally:
            nkv.nkv_set_key_passes("auto")
        assert nkv.nkv_last_device_status(ws) == nkv.NKV_OK, (case, N, d, dtype, H, layers, r, mode)
        rep = pr.SwapReport()
        for g in range(K.shape[0]):
            pr.check_group_against_oracle(K, V, res, g, r, p, rep)
        swaps += rep.swapped_tokens
        heads += rep.heads
    assert swaps <= max(4, heads // 50)


@pytest.mark.gpu
@pytest.mark.parametrize("H,layers,N,d,dtype", [
    (1, 1, 65, 128, "bf16"), (2, 1, 129, 64, "fp16"), (8, 40, 300, 128, "bf16"),   # many heads per SM, spans that cut them
    (3, 1, 6000, 64, "bf16"), (3, 1, 6000, 128, "fp16"),       # blocks of 187 keys
    (2, 1, 7937, 128, "bf16"), (2, 1, 8193, 64, "fp16"),       # a last block of one key
    (1, 1, 40000, 128, "bf16")])                               # every SM starts inside the head
def test_tensor_first_pass_edges(H, layers, N, d, dtype):
    """The tensor-core key passes at the edges of tiles, blocks and the shares of the SMs, against the FMA kernels'
    definition of the same quantities in the oracle (first and last head of the call)."""
    K, _ = _cache(N, d, dtype, H=H, layers=layers)
    p = nkv.nkv_default_params()
    ws = nkv.alloc_workspace(K, p)
    nkv.nkv_set_key_passes("tensor")
    try:
        got = nkv.nkv_key_scan(K, p, ws=ws)
    finally:
        nkv.nkv_set_key_passes("auto")
    assert nkv.nkv_last_device_status(ws) == nkv.NKV_OK
    for g, h in {(0, 0), (layers - 1, H - 1)}:
        ref = oracle.score_head(K[g, h].cpu())
        inv_norm, mu_s, mu_e, a_raw, minmax = (x[g, h].cpu().numpy() for x in got)
        pr.assert_close(inv_norm, ref.inv_norm, "inv_norm", 1e-5)
        pr.assert_close(mu_s, ref.mu_s, "mu_s", 1e-5)
        pr.assert_close(mu_e, ref.mu_e, "mu_e", 1e-5)
        pr.assert_close(a_raw, ref.a_raw, "a_raw", 1e-5)
        pr.assert_close(minmax[0::2], ref.lo, "lo", 1e-5)
        pr.assert_close(minmax[1::2], ref.hi, "hi", 1e-5)


@pytest.mark.gpu
@pytest.mark.parametrize("G,H,N,r,ties", [
    (40, 8, 611, 0.75, "none"), (20, 12, 900, 0.5, "none"), (1, 64, 303, 0.5, "many"), (200, 2, 260, 0.9, "none"),
    (150, 64, 120, 0.5, "none"), (150, 16, 130, 0.75, "many"), (1, 1, 5, 0.5, "none"), (3, 8, 40000, 0.75, "dense"), (1, 16, 20000, 0.9, "all"), (1, 7, 26001, 0.6, "none")])
def test_budget_and_select_in_every_layout(G, H, N, r, ties):
    """One, two, four and eight CTAs per group, several heads per CTA, scores in shared memory and not, bins that
    overflow their lists: budgets and positions bit for bit."""
    s = _random_scores(G, H, N, seed=N + G, ties=ties)
    a_star = torch.from_numpy(s).to(DEV)
    ws = torch.zeros(256 + 256 * ((8 * G * H + 255) // 256), dtype=torch.uint8, device=DEV)
    budgets = nkv.nkv_budget(a_star, r, ws=ws)
    assert nkv.nkv_last_device_status(ws) == nkv.NKV_OK
    idx, offs, _ = nkv.nkv_select(a_star, budgets, H * nkv.nkv_keep_per_head(N, r))
    torch.cuda.synchronize()
    for g in {0, G // 2, G - 1}:
        ref = oracle.budget_select(s[g], r)
        assert np.array_equal(budgets[g].cpu().numpy(), ref.budgets)
        assert np.array_equal(offs[g].cpu().numpy(), ref.offsets)
        assert np.array_equal(idx[g].cpu().numpy(), ref.idx)


@pytest.mark.gpu
@pytest.mark.parametrize("layers,H,N,d", [(40, 8, 701, 64), (20, 12, 1100, 64), (2, 8, 30011, 64), (37, 4, 5000, 64)])
def test_score_to_select_in_every_layout(layers, H, N, d):
    """The score side of the fused call, one head per CTA and several."""
    K, V = _cache(N, d, "bf16", H=H, layers=layers)
    p = nkv.nkv_default_params()
    ws = nkv.alloc_workspace(K, p)
    res = nkv.nkv_compress(K, V, 0.75, p, ws=ws, want_a_star=True)
    assert nkv.nkv_last_device_status(ws) == nkv.NKV_OK
    plain = nkv.nkv_compress(K, V, 0.75, p, ws=ws)     # scores in the padded rows of the workspace
    torch.cuda.synchronize()
    assert torch.equal(plain.idx, res.idx) and torch.equal(plain.budgets, res.budgets)
    rep = pr.SwapReport()
    for g in {0, layers - 1}:
        pr.check_group_against_oracle(K, V, res, g, 0.75, p, rep)
    assert rep.swapped_tokens <= max(2, rep.heads)


@pytest.mark.gpu
@pytest.mark.parametrize("safeguard", [0.0, 0.9, 1.0])
@pytest.mark.parametrize("layers,H,N", [(3, 8, 701), (2, 3, 30011), (30, 12, 900)])
def test_safeguard_that_no_head_and_some_head_needs(layers, H, N, safeguard):
    """Heads that compete once, and twice because one came out short of its safeguard."""
    K, V = _cache(N, 64, "bf16", H=H, layers=layers)
    p = nkv.nkv_default_params()
    p.safeguard = safeguard
    ws = nkv.alloc_workspace(K, p)
    res = nkv.nkv_compress(K, V, 0.75, p, ws=ws, want_a_star=True)
    assert nkv.nkv_last_device_status(ws) == nkv.NKV_OK
    n_safe = nkv.nkv_safeguard_count(N, 0.75, p)
    assert int(res.budgets.min()) >= n_safe
    for g in {0, layers - 1}:
        own = oracle.budget_select(res.a_star[g].cpu().numpy(), 0.75, pr.oracle_params(p))
        assert np.array_equal(own.budgets, res.budgets[g].cpu().numpy())
        assert np.array_equal(own.idx, res.idx[g].cpu().numpy())
        if safeguard == 0.9:
            assert (own.budgets == n_safe).any()


@pytest.mark.gpu
@pytest.mark.parametrize("repeat", [False, True])
@pytest.mark.parametrize("layers,H,N", [(1, 8, 16384), (1, 3, 33333), (4, 8, 16701), (8, 8, 25100), (1, 1, 14400)])
def test_score_phase_with_a_head_shared_by_several_ctas(layers, H, N, repeat):
    """Two, four and eight CTAs per head; keys that repeat crowd the bins of the tails."""
    K, V = _cache(N, 64, "bf16", H=H, layers=layers)
    if repeat:
        K = K[:, :, torch.arange(N, device=DEV) % 7].contiguous()
    p = nkv.nkv_default_params()
    ws = nkv.alloc_workspace(K, p)
    res = nkv.nkv_compress(K, V, 0.75, p, ws=ws, want_a_star=True)
    assert nkv.nkv_last_device_status(ws) == nkv.NKV_OK
    for g in {0, layers - 1}:
        if not repeat:   # equal keys: the tails' members are a matter of rounding
            ref = oracle.compress_group(K[g].cpu(), V[g].cpu(), 0.75, pr.oracle_params(p))
            pr.assert_close(res.a_star[g].cpu().numpy(), ref.a_star, "a_star")
        own = oracle.budget_select(res.a_star[g].cpu().numpy(), 0.75, pr.oracle_params(p))
        assert np.array_equal(own.budgets, res.budgets[g].cpu().numpy())
        assert np.array_equal(own.idx, res.idx[g].cpu().numpy())


@pytest.mark.gpu
@pytest.mark.parametrize("layers,chunk,r,pinned", [(5, 1, 0.75, True), (7, 3, 0.75, True), (4, 4, 0.25, True), (3, 2, 0.75, False)])
def test_host_entry_point_with_rows_fetched_in_place_and_copied(layers, chunk, r, pinned):
    """Retained rows of V read from pinned memory, and V copied whole (most rows retained, or memory that the device
    cannot read); chunks that do and do not divide the groups."""
    K, V = _cache(700, 64, "bf16", H=3, layers=layers)
    dev = nkv.nkv_compress(K, V, r)
    torch.cuda.synchronize()
    hold = (lambda t: t.pin_memory()) if pinned else (lambda t: t)
    Kh, Vh = hold(K.cpu()), hold(V.cpu())
    out = nkv.Compressed(*[hold(torch.empty(t.shape, dtype=t.dtype)) for t in
                           (dev.k_out, dev.v_out, dev.idx, dev.head_offsets, dev.budgets)], None)
    staging = torch.empty(nkv.nkv_host_staging_bytes(3, 700, 64, nkv.NKV_BF16, r, chunk), dtype=torch.uint8, device=DEV)
    nkv.nkv_compress_host(Kh, Vh, r, out, staging, chunk)
    size = lambda t: t.numel() * t.element_size()
    in_place = pinned and r >= 0.4
    assert nkv.nkv_host_bytes() == (size(K) + size(out.v_out if in_place else V),
                                    sum(size(t) for t in (out.k_out, out.v_out, out.idx, out.head_offsets, out.budgets)))
    for a, b in ((out.k_out, dev.k_out), (out.v_out, dev.v_out), (out.idx, dev.idx), (out.head_offsets, dev.head_offsets),
                 (out.budgets, dev.budgets)):
        assert torch.equal(a, b.cpu())


def _keys(s):
    """Ordered keys of fp32 scores: larger score, larger key; NaN by its bits, above +inf or (sign set) below -inf."""
    b = np.ascontiguousarray(s, np.float32).view(np.uint32)
    return np.where(b & 0x80000000, ~b, b | 0x80000000).astype(np.int64)


def _select_by_key(s, r, n_safe):
    """Budgets and positions of one group [H, N] in the order (key descending, head, position), safeguard first."""
    H, N = s.shape
    keep = H * nkv.nkv_keep_per_head(N, r)
    key = _keys(s)
    taken = np.zeros((H, N), bool)
    for h in range(H):
        taken[h, np.lexsort((np.arange(N), -key[h]))[:n_safe]] = True
    head, pos = np.divmod(np.arange(H * N), N)
    order = np.lexsort((pos, head, -key.ravel()))
    order = order[~taken.ravel()[order]]
    taken.ravel()[order[:keep - H * n_safe]] = True
    return taken.sum(1), np.concatenate([np.flatnonzero(t) for t in taken])


@pytest.mark.gpu
@pytest.mark.parametrize("G,H,N,r,share", [(2, 3, 700, 0.5, 0.01), (1, 8, 5000, 0.75, 0.1), (1, 2, 6000, 0.9, 0.5),
                                           (1, 4, 30000, 0.5, 0.4), (3, 1, 9000, 0.5, 1.0)])
def test_scores_that_are_not_finite_are_ordered_by_their_bits(G, H, N, r, share):
    """NaN of either sign, infinities and signed zeros among a caller's scores: every budgeted position is written."""
    rng = np.random.default_rng(N)
    s = _random_scores(G, H, N, seed=N, ties="none")
    odd = np.array([0x7fc00000, 0x7fffffff, 0xffc00000, 0xffffffff, 0x7f800000, 0xff800000, 0x80000000, 0, 0x7f7fffff], np.uint32)
    mask = rng.random(s.shape) < share
    s[mask] = rng.choice(odd, mask.sum()).view(np.float32)
    a_star = torch.from_numpy(s).to(DEV)
    ws = torch.zeros(1 << 16, dtype=torch.uint8, device=DEV)
    budgets = nkv.nkv_budget(a_star, r, ws=ws)
    assert nkv.nkv_last_device_status(ws) == nkv.NKV_OK
    idx, offs, _ = nkv.nkv_select(a_star, budgets, H * nkv.nkv_keep_per_head(N, r), ws=ws)
    assert nkv.nkv_last_device_status(ws) == nkv.NKV_OK
    for g in range(G):
        want_b, want_idx = _select_by_key(s[g], r, nkv.nkv_safeguard_count(N, r))
        assert np.array_equal(budgets[g].cpu().numpy(), want_b)
        assert np.array_equal(idx[g].cpu().numpy(), want_idx)


@pytest.mark.gpu
@pytest.mark.parametrize("N,layers,d,r", [(700, 1, 64, 0.5), (5000, 3, 128, 0.75), (12000, 2, 64, 0.5), (30000, 1, 128, 0.75),
                                          (8192, 19, 128, 0.5)])
def test_a_key_that_is_not_finite_leaves_no_position_unwritten(N, layers, d, r):
    """One infinite key makes the scores of its head NaN: the positions are those of the scores' order all the same."""
    K, V = _cache(N, d, "bf16", H=4, layers=layers)
    K[layers - 1, 2, N // 2, 5] = float("inf")
    ws = nkv.alloc_workspace(K)
    out = nkv.alloc_outputs(K, V, r, want_a_star=True)
    out.idx.fill_(-7)
    res = nkv.nkv_compress(K, V, r, ws=ws, out=out)
    assert nkv.nkv_last_device_status(ws) == nkv.NKV_OK
    assert bool(torch.isnan(res.a_star[layers - 1, 2, 4:]).all())
    for g in {0, layers - 1}:
        want_b, want_idx = _select_by_key(res.a_star[g].cpu().numpy(), r, nkv.nkv_safeguard_count(N, r))
        assert np.array_equal(res.budgets[g].cpu().numpy(), want_b)
        assert np.array_equal(res.idx[g].cpu().numpy(), want_idx)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,d,N", [("bf16", 128, 256), ("bf16", 64, 256), ("fp16", 128, 320), ("fp16", 64, 256)])
def test_a_key_that_is_not_finite_stays_inside_its_head(dtype, d, N):
    """Three heads and more per SM in the tensor-core passes: what the last key of one of them is does not reach the others."""
    K, _ = _cache(N, d, dtype, H=8, layers=56)
    bad = K.clone()
    worst = torch.finfo(K.dtype).max if dtype == "bf16" else float("inf")   # bf16: finite, but not its products
    heads = bad.view(-1, N, d)
    heads[0::15, -1, 3], heads[5::15, -1, 3], heads[10::15, -1] = float("inf"), float("nan"), worst
    p = nkv.nkv_default_params()
    ws = nkv.alloc_workspace(K, p)
    nkv.nkv_set_key_passes("tensor")
    try:
        want, got = nkv.nkv_key_scan(K, p, ws=ws), nkv.nkv_key_scan(bad, p, ws=ws)
    finally:
        nkv.nkv_set_key_passes("auto")
    assert nkv.nkv_last_device_status(ws) == nkv.NKV_OK
    clean = torch.arange(8 * 56) % 5 != 0
    for a, b in zip(want, got):
        assert torch.equal(a.flatten(0, 1)[clean], b.flatten(0, 1)[clean])


@pytest.mark.gpu
@pytest.mark.parametrize("G,H,N,r", [(1, 8, 16384, 0.5), (2, 16, 9001, 0.75), (1, 64, 3000, 0.9), (5, 1, 20000, 0.5), (1, 2, 40003, 0.95)])
@pytest.mark.parametrize("kind", ["sliver", "near zero", "above one", "two values", "ties and sliver"])
def test_bins_that_hold_more_scores_than_a_list(G, H, N, r, kind):
    """Scores that crowd one bin of the competition and of the heads' thresholds, down to one, two and three levels below it."""
    rng = np.random.default_rng(N + len(kind))
    s = rng.random((G, H, N)).astype(np.float32)
    if kind == "sliver":             # one bin of 2048 holds them all
        s = (np.float32(0.3) + np.float32(1e-5) * s * rng.uniform(0.3, 1.0, (G, H, 1))).astype(np.float32)
    elif kind == "near zero":        # the lowest bin: every exponent down to the denormals
        s = np.exp2(-140.0 * s - 12.0).astype(np.float32)
    elif kind == "above one":        # and the highest
        s = np.exp2(120.0 * s + 1.0).astype(np.float32)
    elif kind == "two values":
        s = np.where(s < 0.5, np.float32(0.25), np.nextafter(np.float32(0.25), np.float32(1.0))).astype(np.float32)
    else:
        s = np.where(s < 0.6, np.float32(0.7), np.float32(0.7) + np.float32(1e-6) * rng.integers(-40, 40, s.shape)).astype(np.float32)
    s[:, :, :4] = np.inf
    a_star = torch.from_numpy(s).to(DEV)
    ws = torch.zeros(1 << 20, dtype=torch.uint8, device=DEV)
    budgets = nkv.nkv_budget(a_star, r, ws=ws)
    assert nkv.nkv_last_device_status(ws) == nkv.NKV_OK
    idx, _, _ = nkv.nkv_select(a_star, budgets, H * nkv.nkv_keep_per_head(N, r), ws=ws)
    assert nkv.nkv_last_device_status(ws) == nkv.NKV_OK
    for g in {0, G - 1}:
        want_b, want_idx = _select_by_key(s[g], r, nkv.nkv_safeguard_count(N, r))
        assert np.array_equal(budgets[g].cpu().numpy(), want_b)
        assert np.array_equal(idx[g].cpu().numpy(), want_idx)


@pytest.mark.gpu
@pytest.mark.parametrize("layers,H,N", [(1, 8, 777), (36, 8, 2500), (1, 8, 30011), (20, 8, 9000), (1, 3, 16700)])
def test_keys_whose_anomalies_crowd_a_few_bins(layers, H, N):
    """A head's bulk within a hundredth of the range that a few outliers span: crowded tails of the three scales (one CTA per
    head and several) and a crowded competition."""
    gen = torch.Generator(device=DEV).manual_seed(N)
    mu = 2.0 * torch.randn((layers, H, 1, 64), generator=gen, device=DEV)
    x = mu + 0.05 * torch.randn((layers, H, N, 64), generator=gen, device=DEV)
    # Outliers in every head: the range of an anomaly is then of order 1 and its error of about 1e-7 stays one.  (The bulk by
    # itself spans (0.05 / 2)^2, about 6e-4, and would turn the same error into 2e-4 of a normalised score.)
    outlier = torch.rand((layers, H, N, 1), generator=gen, device=DEV) < 0.002
    outlier[:, :, 10::250] = True
    K = torch.where(outlier, 3.0 * torch.randn(x.shape, generator=gen, device=DEV), x).to(torch.bfloat16)
    p = nkv.nkv_default_params()
    ws = nkv.alloc_workspace(K, p)
    res = nkv.nkv_compress(K, K, 0.5, p, ws=ws, want_a_star=True)
    assert nkv.nkv_last_device_status(ws) == nkv.NKV_OK
    for g in {0, layers - 1}:
        for h in {0, H - 1}:
            pr.assert_close(res.a_star[g, h].cpu().numpy(), oracle.score_head(K[g, h].cpu()).a_star, "a_star")
        own = oracle.budget_select(res.a_star[g].cpu().numpy(), 0.5, pr.oracle_params(p))
        assert np.array_equal(own.budgets, res.budgets[g].cpu().numpy())
        assert np.array_equal(own.idx, res.idx[g].cpu().numpy())


@pytest.mark.gpu
def test_host_entry_point_reports_a_device_status_behind_thousands_of_chunks():
    """The status of the last of 4300 one-group steps (chunks of two groups), of the first, and of none."""
    G, H, N, d, r = 4300, 1, 8, 64, 0.5
    K = torch.randn((G, H, N, d), generator=torch.Generator().manual_seed(1)).to(torch.bfloat16).pin_memory()
    k = nkv.nkv_keep_per_head(N, r)
    out = nkv.Compressed(*[torch.empty(shape, dtype=dt).pin_memory() for shape, dt in (
        ((G, H * k, d), K.dtype), ((G, H * k, d), K.dtype), ((G, H * k), torch.int32), ((G, H + 1), torch.int32), ((G, H), torch.int32))], None)
    staging = torch.empty(nkv.nkv_host_staging_bytes(H, N, d, nkv.NKV_BF16, r, 2), dtype=torch.uint8, device=DEV)
    for chunk in (G // 2 - 1, 0):
        nkv.nkv_debug_set("inject_host_status", chunk * 16 + nkv.NKV_ERR_TIMEOUT)
        try:
            with pytest.raises(nkv.NkvError) as e:
                nkv.nkv_compress_host(K, K, r, out, staging, 2)
            assert e.value.status == nkv.NKV_ERR_TIMEOUT
        finally:
            nkv.nkv_debug_set("inject_host_status", 0)
    nkv.nkv_compress_host(K, K, r, out, staging, 2)
    assert int(out.budgets.sum()) == G * H * k


@pytest.mark.gpu
def test_a_call_that_failed_leaves_no_error_for_the_next():
    """A launch that the runtime refuses (the stream's capture has been invalidated, on the host): the call says so, and the
    next one on a stream in order is not blamed for it."""
    import ctypes
    rt = ctypes.CDLL("libcudart.so.12")
    K, V = _cache(200, 64, "bf16", H=2)
    a_star = torch.rand((1, 2, 200), device=DEV)
    budgets = nkv.nkv_budget(a_star, 0.5)
    idx, offs, _ = nkv.nkv_select(a_star, budgets, 200)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    handle = ctypes.c_void_p(side.cuda_stream)
    graph = ctypes.c_void_p()
    K_out, V_out, ws = (torch.empty((1, 200, 64), dtype=K.dtype, device=DEV) for _ in range(3))
    h = nkv.handle()
    kt, vt = nkv._tensor(K), nkv._tensor(V)
    assert rt.cudaStreamBeginCapture(handle, 2) == 0          # relaxed: other streams stay as they are
    try:
        assert rt.cudaStreamSynchronize(handle) != 0           # not allowed while capturing: ends the capture's validity
        status = h.lib.nkv_compact(h.h, ctypes.byref(kt), ctypes.byref(vt), nkv._p(idx), nkv._p(offs), 200, nkv._p(K_out),
                                   nkv._p(V_out), nkv.NKV_OUT_OF_PLACE, nkv._p(ws), ws.numel(), handle)
    finally:
        rt.cudaStreamEndCapture(handle, ctypes.byref(graph))
        rt.cudaGetLastError()
    assert status == nkv.NKV_ERR_CUDA
    again, _, _ = nkv.nkv_select(a_star, budgets, 200)
    torch.cuda.synchronize()
    assert torch.equal(again, idx)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,d", [("fp16", 64), ("fp16", 128), ("bf16", 128)])
def test_anomalies_do_not_depend_on_the_length_of_the_anchors(dtype, d):
    """nkv_score takes cosines: anchors that a caller brings longer (sums instead of means) or shorter give the same anomalies,
    bit for bit where the factor is a power of two."""
    K, _ = _cache(3000, d, dtype, H=4, layers=10)
    p = nkv.nkv_default_params()
    mu_s, mu_e, inv_norm, _ = nkv.nkv_anchors(K, p)
    nkv.nkv_set_key_passes("tensor")
    try:
        raw = lambda f, g: nkv.nkv_score(K, mu_s * f, mu_e * g, inv_norm, p, want_raw=True)[1]
        want = raw(1.0, 1.0)
        for factor in (4096.0, 2.0 ** -20, 2.0 ** 40):
            assert torch.equal(raw(factor, factor), want), factor
        # the anchors' own rounding, 2^-24 each, and the same again in their norms
        assert float((raw(3000.0, 0.3) - want).abs().max()) <= 1e-6
    finally:
        nkv.nkv_set_key_passes("auto")


@pytest.mark.gpu
def test_own_roots_and_quotients_against_64_bits():
    """The Newton steps behind the approximate reciprocal root, over their range and at its floor: 1/||k|| of keys with one
    component (its square is exact), a_c of unit keys along two axes (integers over the root of an integer), and the
    surprise's extremes."""
    rng = np.random.default_rng(5)
    N, H = 256, 40
    p = nkv.nkv_default_params()
    K = np.zeros((1, H, N, 64), np.float32)
    K[..., 3] = np.exp2(rng.uniform(-60.0, 60.0, (1, H, N)))
    K = torch.from_numpy(K).to(torch.bfloat16).to(DEV)
    nkv.nkv_set_key_passes("tensor")
    try:
        inv = nkv.nkv_key_scan(K, p)[0].cpu().numpy().astype(np.float64)
        axis = torch.from_numpy((rng.random((1, H, N)) < rng.uniform(0.05, 0.95, (1, H, 1))).astype(np.int64)).to(DEV)
        E = torch.nn.functional.one_hot(axis, 64).to(torch.bfloat16)
        a_c = nkv.nkv_key_scan(E, p)[3][0, :, 2].cpu().numpy().astype(np.float64)
    finally:
        nkv.nkv_set_key_passes("auto")
    norm = K[..., 3].double().cpu().numpy()
    # 2^-24 for each of the two roundings behind the last Newton step, and as much again for the floor (1e-24 in fp32)
    assert np.abs(inv * np.maximum(norm, 1e-12) - 1.0).max() <= 2.0 ** -22
    ax = axis[0].cpu().numpy()
    for h in range(H):
        ones = np.concatenate([[0], np.cumsum(ax[h])])
        end = np.arange(1, N + 1)
        beg = np.maximum(0, end - 64)
        n1 = ones[end] - ones[beg]
        n0 = (end - beg) - n1
        want = -np.where(ax[h] == 1, n1, n0) / np.sqrt(n0.astype(np.float64) ** 2 + n1.astype(np.float64) ** 2)
        assert np.abs(a_c[h] / want - 1.0).max() <= 2.0 ** -21   # root and quotient, each corrected once
    C, _ = _cache(2000, 64, "bf16", H=4, layers=10)
    mu_s, mu_e, inv_norm, _ = nkv.nkv_anchors(C, p)
    _, raw, stats = nkv.nkv_score(C, mu_s, mu_e, inv_norm, p, want_raw=True, want_stats=True)
    raw, stats = raw.double().cpu().numpy(), stats.double().cpu().numpy()
    lo, hi = raw.min(-1, keepdims=True), raw.max(-1, keepdims=True)
    s = ((raw - lo) / (hi - lo)).std(2)
    # three normalised values, each within 2^-22 of its own (difference, reciprocal of the range, product); a deviation moves
    # by no more than they do, and the arithmetic behind adds 2^-23
    assert np.abs(stats[..., 12] - s.min(-1)).max() <= 2.0 ** -21 and np.abs(stats[..., 13] - s.max(-1)).max() <= 2.0 ** -21


@pytest.mark.parametrize("N,d,layers", [(128, 128, 1), (129, 64, 1), (1000, 64, 2), (4133, 128, 2), (6000, 64, 1), (6000, 128, 1),
                                        (8193, 128, 1), (8320, 64, 1)] +
                         [(N, d, 43) for N in (4096, 4133, 6000, 8193) for d in (64, 128)])
def test_block_sums_of_the_tensor_pass(N, d, layers):
    """Means of normalised keys whose norms span many powers of two (zero keys among them), against 64 bits.  Blocks that
    end inside a tile, on its edge and after one key.  A sum of 32 terms in tensor memory may lose 2**-24 of its largest
    term per addition and the few additions behind it as much of the sum, so a mean is off by less than 44 * 2**-24 of
    the largest component (the root mean square, as of the FMA form, is 4e-8 of a component's)."""
    g = torch.Generator().manual_seed(N + d)
    K = torch.randn((layers, 3, N, d), generator=g) + 2.0 * torch.randn((layers, 3, 1, d), generator=g)
    K *= torch.exp(3.0 * torch.randn((layers, 3, N, 1), generator=g))
    K[:, :, ::37] = 0
    K = K.to(torch.bfloat16).to(DEV)
    p = nkv.nkv_default_params()
    nkv.nkv_set_key_passes("tensor")
    try:
        _, mu_s, mu_e, _, _ = nkv.nkv_key_scan(K, p)
        torch.cuda.synchronize()
    finally:
        nkv.nkv_set_key_passes("auto")
    k = K.double()
    k = k / k.norm(dim=3, keepdim=True).clamp(min=1e-12)
    b = nkv.nkv_block_size(N, p)
    if layers > 2:   # a CTA goes from block to block and from head to head, 128 keys a block (4096) and odd numbers of them
        assert layers * 3 * nkv.nkv_num_blocks(N, p) > 20 * torch.cuda.get_device_properties(DEV).multi_processor_count
    want = torch.stack([k[:, :, i:i + b].mean(2) for i in range(0, N, b)], 2)
    err = mu_e.double() - want
    assert err.abs().max() <= 44 * 2.0 ** -24 * k.abs().max()
    assert err.square().mean().sqrt() <= 2e-7 * want.square().mean().sqrt()
    assert (mu_s.double() - k.mean(2)).abs().max() <= 44 * 2.0 ** -24 * k.abs().max()


@pytest.mark.parametrize("layers,H,N,r,kind", [(1, 1, 130, 0.5, "plain"), (2, 3, 777, 0.5, "plain"), (1, 5, 2049, 0.75, "plain"),
                                               (1, 33, 515, 0.85, "plain"), (1, 64, 300, 0.25, "plain"), (3, 8, 4097, 0.95, "plain"),
                                               (1, 8, 6000, 0.75, "crowded"), (2, 7, 1030, 0.5, "equal"), (1, 4, 2500, 0.75, "short")])
def test_fused_competition_matches_the_budget_call(layers, H, N, r, kind):
    """The fused call takes the pool's bin from the histograms that the scores left; nkv_budget and nkv_select work on the
    scores alone.  Same scores, same integers: heads in any number, bins that hold most scores, scores all equal, and a
    head that only its safeguard keeps."""
    K, V = _cache(N, 64, "bf16", H=H, layers=layers, seed=5 + N)
    if kind == "crowded":
        K = (K[:, :, :1] + 0.02 * K).contiguous()
    elif kind == "equal":
        K = K[:, :, :1].expand_as(K).contiguous()
    elif kind == "short":
        K[:, 1] = (K[:, 1, :1] + 0.001 * K[:, 1].float()).to(K.dtype)
    p = nkv.nkv_default_params()
    ws = nkv.alloc_workspace(K, p)
    res = nkv.nkv_compress(K, V, r, p, ws=ws, want_a_star=True)
    assert nkv.nkv_last_device_status(ws) == nkv.NKV_OK
    budgets = nkv.nkv_budget(res.a_star, r, p)
    idx, offs, _ = nkv.nkv_select(res.a_star, budgets, res.idx.shape[1])
    assert torch.equal(res.budgets, budgets)
    assert torch.equal(res.head_offsets, offs)
    assert torch.equal(res.idx, idx)


def _crowded_keys(layers, H, N):
    """Keys whose scores lie in the lowest bin of 2048 but for some outliers, unevenly over the heads."""
    gen = torch.Generator().manual_seed(N)
    x = 2.0 * torch.randn((layers, H, 1, 64), generator=gen) + 0.05 * torch.randn((layers, H, N, 64), generator=gen)
    outlier = torch.rand((layers, H, N, 1), generator=gen) < 0.002
    outlier[:, :, 10::250] = True
    return torch.where(outlier, 3.0 * torch.randn(x.shape, generator=gen), x).to(torch.bfloat16).to(DEV)


@pytest.mark.parametrize("layers,H,N", [(1, 8, 30011), (20, 8, 9000), (1, 8, 4096), (1, 5, 9000), (1, 3, 16700)])
def test_crowded_competition_again_and_again(layers, H, N):
    """The heads' counts of a crowded bin come from the CTAs that have the heads.  A hundred calls, each against the budget
    and the select call on the same scores; the bin that holds the last slot has more scores than any list, and in most groups no head
    comes out short of its safeguard, so that one attempt settles it."""
    r = 0.5
    K = _crowded_keys(layers, H, N)
    p = nkv.nkv_default_params()
    ws = nkv.alloc_workspace(K, p)
    for call in range(100):
        res = nkv.nkv_compress(K, K, r, p, ws=ws, want_a_star=True)
        assert nkv.nkv_last_device_status(ws) == nkv.NKV_OK
        budgets = nkv.nkv_budget(res.a_star, r, p)
        idx, offs, _ = nkv.nkv_select(res.a_star, budgets, res.idx.shape[1])
        assert torch.equal(res.budgets, budgets) and torch.equal(res.head_offsets, offs) and torch.equal(res.idx, idx)
        if call == 0:
            keep = res.idx.shape[1]
            for g in {0, layers - 1}:
                s = res.a_star[g].double().clamp(max=1.0)
                bins = (s * 2047).round()
                inside = bins == bins.flatten().topk(keep).values[-1]
                assert int(inside.sum()) > 6144 and s[inside].unique().numel() > 6144
                own = oracle.budget_select(res.a_star[g].cpu().numpy(), r, pr.oracle_params(p))
                assert np.array_equal(own.budgets, res.budgets[g].cpu().numpy()) and np.array_equal(own.idx, res.idx[g].cpu().numpy())
            assert 2 * int((res.budgets.min(1).values > nkv.nkv_safeguard_count(N, r, p)).sum()) > layers


@pytest.mark.parametrize("G,H,N", [(1, 1, 700), (2, 2, 900), (1, 3, 700), (1, 5, 5000), (3, 8, 2049), (1, 8, 32768), (2, 12, 3001), (1, 64, 400)])
def test_budget_of_heads_short_of_their_safeguard(G, H, N):
    """Heads that come out short for certain (none of their scores reaches the bin of the last slot), that fall short by the
    scores inside that bin, and that have just enough: budgets bit for bit."""
    r = 0.75
    rng = np.random.default_rng(N + H)
    s = rng.random((G, H, N)).astype(np.float32)
    n_safe = nkv.nkv_safeguard_count(N, r)
    if H > 1:
        s[:, 0] *= np.float32(0.25)               # nothing near the others' best
        for h in range(1, H, 3):                  # its n_safe best, one more and one less, around the others' quarter
            top = n_safe - 5 + (h // 3) % 3       # (and four sinks)
            s[:, h] = np.float32(0.3) * rng.random((G, N)).astype(np.float32)
            s[:, h, 5:5 + top] = np.float32(0.999)
    s[:, :, :4] = np.inf
    a_star = torch.from_numpy(s).to(DEV)
    ws = torch.zeros(1 << 16, dtype=torch.uint8, device=DEV)
    budgets = nkv.nkv_budget(a_star, r, ws=ws)
    assert nkv.nkv_last_device_status(ws) == nkv.NKV_OK
    for g in range(G):
        assert np.array_equal(budgets[g].cpu().numpy(), _select_by_key(s[g], r, n_safe)[0])
    if H > 3:   # (of fewer heads too many are low)
        assert int(budgets[:, 0].max()) == n_safe


class _Kind(torch.Tensor):
    pass


@pytest.mark.filterwarnings("ignore:Named tensors")
def test_caches_of_a_subclass_and_with_named_dimensions():
    K, V = _cache(300, 64, "bf16", H=3)
    want = nkv.nkv_compress(K, V, 0.5)
    names = ("g", "h", "n", "d")
    for k, v in ((K.as_subclass(_Kind), V.as_subclass(_Kind)), (K.refine_names(*names), V.refine_names(*names))):
        got = nkv.nkv_compress(k, v, 0.5)
        for name in ("k_out", "v_out", "idx", "head_offsets", "budgets"):
            t = getattr(got, name)
            assert type(t) is torch.Tensor and torch.equal(t, getattr(want, name))
