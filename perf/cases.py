"""Workloads of the decode path, run through its public entry points.

A case is one call (or one token) of a program that decodes with this package:

* ``step``     one token through ``np_step``: predictor, selection, delta, transfer of the incoming rows
               from the pinned record store and the MLP chain, with the residency the earlier tokens left.
* ``select``   one token with the centroid selection: ``np_trunk_forward``, ``np_centroid_select``,
               ``np_step_selected``.
* ``predict``  ``np_predict`` with the logits and the bitmap handed out (a caller that plans residency itself).
* ``chain``    ``np_mlp_chain`` over rows that are resident already (a stack whose rows stay on the GPU, or
               the last token again with another input).

Shapes are those of ``synth.CONFIGS``; the record store is aliased over a few layers
(``store_layers``), which leaves row counts and traffic as they are and keeps the set-up short.
Weights and hidden states are drawn as in ``synth``: ``randn * 0.02`` in bf16 and an AR(1) sequence
of hidden states.
"""
import math

import torch

from paper_2608_22643_b200 import binding as nb
from paper_2608_22643_b200 import synth

TOKENS = 64       # hidden states a decoding case walks through, forth and back (the AR(1) overlap holds both ways)
WARM_TOKENS = 3   # tokens decoded before the first pass: the cold start is not the steady state

TRANSFER = {"runs": nb.NP_XFER_MEMCPY_RUNS, "gather": nb.NP_XFER_HOST_GATHER, "zerocopy": nb.NP_XFER_ZERO_COPY}
POLICY = {"exact": nb.NP_EVICT_EXACT, "lru": nb.NP_EVICT_LRU}
RECORDS = {"bf16": nb.NP_REC_BF16, "int8": nb.NP_REC_INT8}

# the paper's predictor: T, K, K0, E and the number of trunk blocks
TRUNK_T, TRUNK_K, TRUNK_K0, TRUNK_E, TRUNK_BLOCKS = 512, 512, 512, 2048, 4


def _case(path, shape, **kw):
    c = {"path": path, "L": shape.n_layers, "D": shape.d_model, "M": shape.d_ffn, "H": shape.d_pred,
         "k": shape.top_k, "C": shape.capacity, "B": 1, "rho": shape.rho, "policy": "exact",
         "transfer": "gather", "records": "bf16", "dense": 0, "store_layers": min(4, shape.n_layers)}
    c.update(kw)
    return c


def listed():
    tiny, s7, s13, s70 = (synth.CONFIGS[n] for n in ("tiny", "7b", "13b", "70b"))
    return [
        # the smallest stack, one token with the configuration defaults: launches and latency
        _case("step", tiny, name="step tiny", transfer="runs"),
        # one sequence decoding with the 7B-shaped stack: the ordinary use, bound by the transfer of the rows
        _case("step", s7, name="step 7b"),
        # the same for the 13B-shaped stack with rows kept while capacity allows
        _case("step", s13, name="step 13b lru", policy="lru"),
        # sixteen sequences per step over the union of their rows
        _case("step", s7, name="step 7b x16", B=16),
        # a memory budget that holds three quarters of the layers whole, and 8-bit records for the others
        _case("step", s7, name="step 7b dense24 int8", dense=24, records="int8"),
        # the paper's own predictor and centroid selection in front of the same path
        _case("select", s7, name="select 7b"),
        # scores and sets of all layers for one sequence: a pass over the predictor's weights
        _case("predict", s7, name="predict 7b"),
        # a small odd batch
        _case("predict", s13, name="predict 13b x3", B=3),
        # a full batch
        _case("predict", s7, name="predict 7b x16", B=16),
        # the MLP stack over resident rows, one sequence
        _case("chain", s7, name="chain 7b", store_layers=1),
        # sixteen sequences
        _case("chain", s7, name="chain 7b x16", B=16, store_layers=1),
        # the largest stack
        _case("chain", s70, name="chain 70b", store_layers=1),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the same ranges: widths from 256 to 8192, 2 to 80 layers, 1 to 16 sequences."""
    path = rng.choice(["step", "step", "step", "select", "predict", "predict", "chain", "chain", "chain"])
    grain = rng.choice([64, 64, 64, 16])                       # widths are multiples of 64, some ragged
    D = max(256, int(_log_uniform(rng, 256, 8192)) // grain * grain)
    M = int(D * rng.uniform(2.5, 4.0)) // 32 * 32
    h_grain = rng.choice([64, 64, 64, 8])
    H = min(1024, max(64, int(D / rng.uniform(5, 9)) // h_grain * h_grain))
    L = int(_log_uniform(rng, 2, 80))
    B = 1 if path == "select" else rng.choice([1, 1, 1, 1, 2, 3, 4, 6, 8, 11, 16, 16])
    k = max(1, int(M * rng.uniform(0.04, 0.12 if B == 1 else 0.1)))
    C = int(M * rng.uniform(0.25, 0.4)) if B > 1 else max(k, int(M * rng.uniform(0.15, 0.4)))
    # no more rows, predictor weights or resident bytes than the largest listed case has
    L = max(2, min(L, int(5.0e9 / (6 * D * k * min(B, 2.2))), int(4.5e9 / (2 * M * H)), int(20e9 / (6 * D * C))))
    if path == "step":      # a token's transfer stays near the 13B-shaped one
        L = max(2, min(L, int(1.2e9 / (6 * D * k * min(B, 2.2)))))
    dense = 0
    if path in ("step", "chain") and D % 256 == 0 and rng.random() < 0.2:
        dense = max(1, min(L - 1, int(rng.uniform(0.2, 0.8) * L), int(6e9 / (6 * D * M))))
    records = "int8" if path == "step" and rng.random() < 0.2 else "bf16"
    transfer = rng.choice(["gather", "gather", "zerocopy", "runs"]) if path == "step" else "gather"
    if transfer == "runs":  # one copy call per run of rows: small stacks only
        L = max(2, min(L, 6000 // k))
        dense = min(dense, L - 1)
    return {"path": path, "L": L, "D": D, "M": M, "H": H, "k": k, "C": C, "B": B,
            "rho": rng.choice([0.9, 0.95, 0.97, 0.97, 0.985]), "policy": rng.choice(["exact", "exact", "lru"]),
            "transfer": transfer, "records": records, "dense": dense,
            "store_layers": min(L, 1 if path == "chain" else 2)}


def _stack(c, seed):
    return synth.StackConfig("case", c["L"], c["D"], c["M"], c["H"], 0, 0, TOKENS, seed, c["rho"])


def _store(cfg, c):
    """The record blocks of the first ``store_layers`` layers in pinned host memory, bf16 or 8-bit."""
    n = c["store_layers"]
    shape = (n, cfg.d_ffn, 3, cfg.d_model)
    if c["records"] == "bf16":
        out = torch.empty(shape, dtype=torch.bfloat16, pin_memory=True)
        return synth.fill_backing_store(cfg.with_(n_layers=n), out, "cuda")
    full = torch.empty(shape, dtype=torch.bfloat16, device="cuda")
    synth.fill_backing_store(cfg.with_(n_layers=n), full, "cuda")
    out = torch.empty((n, cfg.d_ffn, 3 * cfg.d_model + 16), dtype=torch.uint8, pin_memory=True)
    return synth.quantize_store(full, device="cuda", out=out)


def _centroid_bank(cfg, k, generator):
    """``synth.centroid_bank`` drawn on the GPU: masks of k neurons, popularity plus per-centroid noise."""
    L, M, K = cfg.n_layers, cfg.d_ffn, TRUNK_K
    bank = torch.empty((L, 2, K, M // 32), dtype=torch.int32, device="cuda")
    weights = (1 << torch.arange(32, dtype=torch.int64, device="cuda"))
    for l in range(L):
        pop = torch.randn(M, generator=generator, device="cuda")
        for h in range(2):
            score = pop[None, :] + torch.randn(K, M, generator=generator, device="cuda")
            bits = torch.zeros((K, M), dtype=torch.int64, device="cuda")
            bits.scatter_(1, score.topk(k, dim=1).indices, 1)
            bank[l, h] = (bits.view(K, M // 32, 32) * weights).sum(dim=2).to(torch.int32)
    return bank


def _trunk(state, cfg, c, seed):
    """The predictor's weights, bank and per-token features, derived from the hidden states."""
    L, D = c["L"], c["D"]
    gen = torch.Generator(device="cuda").manual_seed(seed + 99)
    dims = (D, D, 128, 1)
    w = synth.trunk_weights(TRUNK_T, dims, TRUNK_K0, TRUNK_E, TRUNK_BLOCKS, 1, TRUNK_K, seed, device="cuda")
    heads = torch.randn(L * 2 * TRUNK_K, 8 * TRUNK_T, generator=gen, device="cuda")
    w["heads"] = (heads * (8 * TRUNK_T) ** -0.5).to(torch.bfloat16)
    desc, table = nb.trunk_pack(w, L)
    x = state["x"][:, 0].to(torch.float32)
    proj = torch.randn(D, TRUNK_K0, generator=gen, device="cuda") / D ** 0.5
    rms = torch.cat([x.pow(2).mean(dim=1, keepdim=True).sqrt(), torch.zeros(TOKENS, 7, device="cuda")], dim=1)
    feats = [x.contiguous(), torch.nn.functional.layer_norm(x, (D,)).contiguous(), x[:, :128].contiguous(), rms]
    ids = (x @ proj).argmax(dim=1).to(torch.int32)
    state.update(
        trunk=(desc, table), weights=w, bank=_centroid_bank(cfg, c["k"], gen),
        features=[([f[t] for f in feats], ids[t:t + 1]) for t in range(TOKENS)],
        work=torch.empty(nb.np_trunk_workspace_floats(desc), dtype=torch.float32, device="cuda"),
        head_logits=torch.empty((1, L, 2, TRUNK_K), dtype=torch.float32, device="cuda"),
        ids=torch.empty((1, L, 2), dtype=torch.int32, device="cuda"),
        bitmap=torch.empty((L, c["M"] // 32), dtype=torch.int32, device="cuda"))


def _engine(c, cfg):
    w1, w2 = synth.predictor_weights(cfg, "cuda")
    ncfg = nb.make_config(c["L"], c["D"], c["M"], c["H"], c["k"], c["C"], max_batch=c["B"],
                          evict_policy=POLICY[c["policy"]], transfer_mode=TRANSFER[c["transfer"]],
                          record_format=RECORDS[c["records"]], dense_layers=c["dense"],
                          store_layers=c["store_layers"])
    return nb.Engine(ncfg, w1, w2, _store(cfg, c))


def _token(s):
    """The next hidden state's index: 0 1 .. T-1 T-2 .. 1 0 1 .."""
    t = s["t"] % (2 * TOKENS - 2)
    s["t"] += 1
    return t if t < TOKENS else 2 * TOKENS - 2 - t


def _decode(s):
    """One token: what a decoding program calls."""
    e, t = s["engine"], _token(s)
    if s["case"]["path"] == "select":
        feats, cid = s["features"][t]
        nb.np_trunk_forward(*s["trunk"], feats, cid, s["work"], s["head_logits"], e.stream)
        nb.np_centroid_select(e.ctx, s["head_logits"], 1, TRUNK_K, s["bank"], s["ids"], s["bitmap"], e.stream)
        nb.np_step_selected(e.ctx, s["tokens"][t], 1, s["bitmap"], s["out"], e.stream, e.copy_stream)
    else:
        nb.np_step(e.ctx, s["tokens"][t], s["case"]["B"], s["out"], e.stream, e.copy_stream)


def prepare(case, seed):
    cfg = _stack(case, seed)
    B, L, D, M = case["B"], case["L"], case["D"], case["M"]
    s = {"case": case, "t": 0, "engine": _engine(case, cfg),
         "x": synth.hidden_states(cfg, TOKENS, batch=B).to("cuda"),
         "out": torch.empty((B, D), dtype=torch.float32, device="cuda")}
    s["tokens"] = [s["x"][t] for t in range(TOKENS)]
    if case["path"] == "predict":
        s["logits"] = torch.empty((B, L, M), dtype=torch.float32, device="cuda")
        s["bitmap"] = torch.empty((L, M // 32), dtype=torch.int32, device="cuda")
    if case["path"] == "select":
        _trunk(s, cfg, case, seed)
    torch.cuda.synchronize()
    if case["path"] == "chain":
        _decode(s)
    elif case["path"] != "predict":
        for _ in range(WARM_TOKENS):
            _decode(s)
    torch.cuda.synchronize()
    return s


def run(s):
    c, e = s["case"], s["engine"]
    if c["path"] == "predict":
        nb.np_predict(e.ctx, s["tokens"][_token(s)], c["B"], s["logits"], s["bitmap"], e.stream)
        return {"logits": s["logits"], "bitmap": s["bitmap"]}
    if c["path"] == "chain":
        nb.np_mlp_chain(e.ctx, s["tokens"][_token(s)], c["B"], s["out"], e.stream)
        return s["out"]
    _decode(s)
    if c["path"] == "select":
        return {"out": s["out"], "head_logits": s["head_logits"], "ids": s["ids"], "bitmap": s["bitmap"]}
    if c["B"] == 1:   # the updated row buffers; a batch's sets may differ by a row (see tolerance)
        return {"out": s["out"], "gate": e.gate, "up": e.up, "downT": e.downT}
    return s["out"]


def _rows(c):
    """Rows of a layer that one pass uses (the union over a batch), and how many of them are new to it."""
    used = c["k"] * (1 + 0.28 * math.log2(c["B"]))
    if c["path"] == "select":
        used *= 0.32                              # gate AND up
    used = min(used, c["C"])
    new = used * 0.95 * math.sqrt(1 - c["rho"])   # what an AR(1) sequence of this rho replaces
    if c["B"] > 1:
        new *= 0.75
    if c["policy"] == "lru":
        new *= 0.35
    return used, new


def work(case):
    c = case
    B, L, D, M, H, nd = c["B"], c["L"], c["D"], c["M"], c["H"], c["dense"]
    record = 6 * D
    used, new = _rows(c)
    predict = {"bytes": 2 * H * D + 2 * (L - nd) * M * H + 2 * B * D + (L - nd) * M / 8,
               "flops": 2 * B * (H * D + (L - nd) * M * H)}
    if c["path"] == "select":
        params = 2 * TRUNK_T * D + 5 * TRUNK_T * TRUNK_E + 64 * TRUNK_BLOCKS * TRUNK_T ** 2 + 16 * L * TRUNK_K * TRUNK_T
        predict = {"bytes": 2 * params + L * M / 4, "flops": 2 * params}
    if c["path"] == "predict":
        return {"bytes": predict["bytes"] + 4 * B * L * M, "flops": predict["flops"]}
    rows = nd * M + (L - nd) * used
    chain = {"bytes": rows * record + 6 * B * D, "flops": 6 * B * D * rows}
    if c["path"] == "chain":
        return chain
    stored = 3 * D + 16 if c["records"] == "int8" else record
    moved = (L - nd) * new * (stored + record)
    return {"bytes": predict["bytes"] + chain["bytes"] + moved, "flops": predict["flops"] + chain["flops"]}


def tolerance(case):
    """About four times what other summation orders of the same products show.

    Measured with the kernels for comparison runs (plain cores in place of tensor cores, rows dealt in
    another way): logits differ by 5e-7 (2.4e-6 at most), the chain by 1e-6 to 2.6e-6 (1.1e-5 at most),
    row buffers not at all.  A batch makes B * L selections per token, and every few tokens one of them is
    decided by less than the logits' rounding: a step's result then lacks one row of one layer for
    another, which moves it by 1e-3 to 7e-3 (2e-1 at most), measured by exchanging one row.
    """
    if case["path"] == "predict":
        return {"rel": 4e-6, "max": 2e-5, "differ": 1e-3}
    if case["path"] == "step" and case["B"] > 1:
        return {"rel": 1e-2, "max": 2e-1}
    return {"rel": 1e-5, "max": 4e-5, "differ": 1e-3}
