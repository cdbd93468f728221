"""Workloads whose speed counts: KV caches compressed through the public entry points of ``nkv``.

A case is one call (or one chain of stage calls) on a whole cache ``[G, H, N, d]``, G = sequences x layers.
Shapes and eviction ratios are those of ``paper_2605_26678_b200/workloads.py`` and of the tests, at the aligned
lengths that benchmarks use and at the ragged ones that prompts have.

Inputs.  Keys follow the recipe of ``workloads.py`` (a mean direction per head, segments with offsets, unit noise,
needles that leave the mean direction, sink rows scaled by eight; values N(0, 1)), drawn with the device's own
generator.  One thing is set differently: a layer holds as many needles as it has slots left beside its sinks, spread
unevenly over its heads.  The retained set is then the needles and the sinks whatever the order of summation in the
scores.  With the recipe's 0.1 % of needles the scores around a layer's threshold lie about 1e-6 apart, so two correct
implementations swap a few near ties, and one swap shifts every packed row behind it: the outputs of a pass could not
be compared.  The budgets still differ from head to head, and the scores on either side of the threshold are as
continuous as before.
"""
import math

import torch

from paper_2605_26678_b200 import nkv

_DTYPES = {"bf16": torch.bfloat16, "fp16": torch.float16, "fp32": torch.float32}
_SINKS = 4
_MAX_BYTES = 2 * 144 * 8 * 32768 * 128 * 2     # K + V of the largest listed case
_MAX_KEYS = 144 * 8 * 32768


def _case(name, layers, batch, n, d, dtype, r, path="compress", heads=8):
    c = {"layers": layers, "batch": batch, "heads": heads, "n": n, "d": d, "dtype": dtype, "r": r, "path": path}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a short prompt, one layer as soon as its prefill is done, called as the README shows it (nothing kept between calls)
        _case("layer_short_bf16", 1, 1, 777, 128, "bf16", 0.5, "plain"),
        # the single-layer fp32 configuration
        _case("layer_4k_fp32", 1, 1, 4096, 128, "fp32", 0.75),
        # layer by layer compression during the prefill of a long prompt
        _case("layer_32k_bf16", 1, 1, 32768, 128, "bf16", 0.75),
        # a chat-sized prompt on the Llama-3.2-1B shape, ragged length
        _case("llama1b_2k", 16, 1, 2500, 64, "bf16", 0.5),
        # the usual ragged prompt between 4k and 8k (its episodic blocks are not a multiple of eight keys)
        _case("qwen4b_6k_ragged", 36, 1, 6000, 128, "bf16", 0.75),
        # the benchmark's 8k, 32k (d = 64), 32k x 4 and 128k configurations
        _case("qwen4b_8k", 36, 1, 8192, 128, "bf16", 0.75),
        _case("llama1b_32k", 16, 1, 32768, 64, "bf16", 0.95),
        _case("qwen4b_32k_b4", 36, 4, 32768, 128, "bf16", 0.75),
        _case("qwen8b_128k", 36, 1, 131072, 128, "bf16", 0.95),
        # a cache stored in fp16, light eviction
        _case("qwen8b_16k_fp16", 36, 1, 16384, 128, "fp16", 0.5),
        # the stages one by one, every intermediate in the caller's hands
        _case("staged_qwen06b_4k", 28, 1, 4133, 128, "bf16", 0.75, "staged"),
        # a cache that was offloaded to pinned host memory
        _case("host_llama1b_8k", 16, 1, 8192, 64, "bf16", 0.75, "host"),
    ]


def draw(rng):
    layers, d = rng.choice([(1, 128), (1, 64), (2, 128), (4, 128), (16, 64), (28, 128), (36, 128), (36, 128), (64, 128)])
    batch = rng.choice([1, 1, 1, 2, 4])
    heads = rng.choice([8, 8, 8, 4, 2])
    dtype = rng.choice(["bf16", "bf16", "bf16", "bf16", "fp16", "fp32"])
    # the lightest eviction only where a direction has enough channels to tell a needle from the rest by
    r = rng.choice([0.25 if d == 128 else 0.5, 0.5, 0.75, 0.75, 0.85, 0.95])
    path = rng.choice(["compress"] * 7 + ["plain", "staged", "host"])
    eb = 4 if dtype == "fp32" else 2
    most = {"staged": 3_000_000, "host": 2_500_000}.get(path, _MAX_KEYS)
    units = layers * batch * heads
    hi = min(131072, most // units, _MAX_BYTES // (2 * units * d * eb))
    n = int(round(math.exp(rng.uniform(math.log(512), math.log(max(hi, 600))))))
    if rng.random() < 0.4:     # the lengths that contexts are cut to
        n = max(512, n // 256 * 256)
    return _case(None, layers, batch, n, d, dtype, r, path, heads)


def _needle_mask(gen, H, N, k, r, device):
    """[H, N] bool: H * (k - sinks) needle rows behind the sinks, evenly mixed with the others.  A head holds more or less
    than its share by up to 40 % (less when most of the cache is kept, so that every head has rows to drop)."""
    m = k - _SINKS
    spread = 0.4 * min(1.0, r / 0.75) ** 2
    share = 1.0 - spread + 2.0 * spread * torch.rand(H, generator=gen, device=device, dtype=torch.float64)
    count = (share * (m * H / share.sum())).floor().clamp(max=N - _SINKS)
    # what rounding and the clamp left over goes to the heads that have room, in order
    left = H * m - count.sum()
    room = (N - _SINKS) - count
    before = torch.cumsum(room, 0) - room
    count += torch.minimum((left - before).clamp(min=0), room)
    phase = torch.arange(N - _SINKS, device=device) * 0.6180339887498949 + torch.rand((H, 1), generator=gen, device=device,
                                                                                      dtype=torch.float64)
    jitter = 0.1 * torch.rand((H, N - _SINKS), generator=gen, device=device)
    key = phase % 1.0 + jitter
    # no needles among the last rows: the last episodic block may be a handful of keys, and their mean has to be theirs
    key[:, -32:] += 2.0
    order = key.argsort(1)
    mask = torch.zeros((H, N), dtype=torch.bool, device=device)
    picked = torch.arange(N - _SINKS, device=device).unsqueeze(0) < count.unsqueeze(1)
    mask[:, _SINKS:].scatter_(1, order, picked)
    return mask


def _fill_group(gen, K, V, k, r):
    """One group [H, N, d] of the cache."""
    H, N, d = K.shape
    dev = K.device
    seg_lo, seg_hi = min(256, N), min(2048, 2 * N)
    mu = 2.0 * torch.randn((H, 1, d), generator=gen, device=dev)
    S = (N + seg_lo - 1) // seg_lo
    ends = torch.randint(seg_lo, seg_hi + 1, (H, S), generator=gen, device=dev).cumsum(1)
    rows = torch.arange(N, device=dev).expand(H, N).contiguous()
    seg = torch.searchsorted(ends, rows, right=True)
    offsets = 0.5 * torch.randn((H, S, d), generator=gen, device=dev)
    x = torch.randn((H, N, d), generator=gen, device=dev)
    mask = _needle_mask(gen, H, N, k, r, dev).unsqueeze(2)
    bulk = mu + torch.gather(offsets, 1, seg.unsqueeze(2).expand(H, N, d))
    x = torch.where(mask, 3.0 * x, bulk + x)
    x[:, :_SINKS] *= 8.0
    K.copy_(x)
    V.copy_(torch.randn((H, N, d), generator=gen, device=dev))


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    G, H, N, d, r = case["layers"] * case["batch"], case["heads"], case["n"], case["d"], case["r"]
    dt = _DTYPES[case["dtype"]]
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    K = torch.empty((G, H, N, d), dtype=dt, device=dev)
    V = torch.empty((G, H, N, d), dtype=dt, device=dev)
    k = nkv.nkv_keep_per_head(N, r)
    for g in range(G):
        _fill_group(gen, K[g], V[g], k, r)
    state = {"path": case["path"], "K": K, "V": V, "r": r, "keep": H * k}
    if case["path"] == "plain":
        return state
    state["params"] = nkv.nkv_default_params()
    if case["path"] == "host":
        # four groups at a time, as bench.py stages them; everything the call reads and writes is pinned
        chunk = min(4, G)
        code = {"bf16": nkv.NKV_BF16, "fp16": nkv.NKV_F16, "fp32": nkv.NKV_F32}[case["dtype"]]
        pin = dict(pin_memory=True)
        hK, hV = torch.empty((G, H, N, d), dtype=dt, **pin), torch.empty((G, H, N, d), dtype=dt, **pin)
        hK.copy_(K)
        hV.copy_(V)
        i32 = dict(dtype=torch.int32, **pin)
        state.update(
            K=hK, V=hV, chunk=chunk,
            staging=torch.empty(nkv.nkv_host_staging_bytes(H, N, d, code, r, chunk, state["params"]), dtype=torch.uint8, device=dev),
            out=nkv.Compressed(torch.empty((G, H * k, d), dtype=dt, **pin), torch.empty((G, H * k, d), dtype=dt, **pin),
                               torch.empty((G, H * k), **i32), torch.empty((G, H + 1), **i32), torch.empty((G, H), **i32), None))
        return state
    state["ws"] = nkv.alloc_workspace(K, state["params"])
    if case["path"] == "compress":
        state["out"] = nkv.alloc_outputs(K, V, r)
    return state


def _outputs(o):
    return {"k_out": o.k_out, "v_out": o.v_out, "idx": o.idx, "head_offsets": o.head_offsets, "budgets": o.budgets}


def run(state):
    K, V, r = state["K"], state["V"], state["r"]
    if state["path"] == "plain":
        return _outputs(nkv.nkv_compress(K, V, r))
    p = state["params"]
    if state["path"] == "host":
        return _outputs(nkv.nkv_compress_host(K, V, r, state["out"], state["staging"], state["chunk"], p))
    ws = state["ws"]
    if state["path"] == "compress":
        return _outputs(nkv.nkv_compress(K, V, r, p, out=state["out"], ws=ws))
    mu_s, mu_e, inv_norm, _ = nkv.nkv_anchors(K, p, ws=ws)
    a_star, _, _ = nkv.nkv_score(K, mu_s, mu_e, inv_norm, p, ws=ws)
    budgets = nkv.nkv_budget(a_star, r, p, ws=ws)
    idx, offs, _ = nkv.nkv_select(a_star, budgets, state["keep"], ws=ws)
    k_out, v_out = nkv.nkv_compact(K, V, idx, offs, ws=ws)
    return {"mu_s": mu_s, "mu_e": mu_e, "inv_norm": inv_norm, "a_star": a_star, "budgets": budgets, "idx": idx,
            "head_offsets": offs, "k_out": k_out, "v_out": v_out}


def work(case):
    """K is read once; the retained rows of K and V are read and written; positions are written.  Operations per key and
    channel: the norm, the running window sum and its two dots, the two anchor dots, the block sum."""
    G, H, N, d = case["layers"] * case["batch"], case["heads"], case["n"], case["d"]
    eb = 4 if case["dtype"] == "fp32" else 2
    keys, kept = G * H * N, G * H * nkv.nkv_keep_per_head(N, case["r"])
    nbytes = keys * d * eb + kept * (4 * d * eb + 4) + G * (2 * H + 1) * 4
    if case["path"] == "staged":   # the scores and reciprocal norms are outputs of their own
        nbytes += keys * 8
    return {"bytes": nbytes, "flops": keys * d * 16}


def tolerance(case):
    # rows are copied verbatim and the retained set does not hinge on rounding (see the module's head): bytes stay
    # the same.  The stage calls also return fp32 anchors, norms and scores.
    return {"rel": 1e-5, "max": 1e-4, "differ": 0.0} if case["path"] == "staged" else "exact"
