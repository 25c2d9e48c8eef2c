"""What a program that serves with this library has it do, as cases that can be timed and compared.

A case is one pass through the public entry points (paper_2511_12934_b200.binding.Aif): a scoring call of one request
or of a batch of requests, with ids and logits in GPU or in host memory; a whole request from raw user features; an
update of the item table.  Sizes are those of the benchmark's workloads (paper_2511_12934_b200.synth), their mini-batches
and the ranges around them; inputs follow the same distributions, drawn on the GPU from the seed.
"""
import math

import torch

from paper_2511_12934_b200 import binding as B
from paper_2511_12934_b200 import synth

# The three model shapes of the benchmark's workloads: the fp32 one, the paper-shaped one and the wide one.
MODELS = {
    "small": dict(dtype=B.F32, d=64, F=8, B=16, dc=16, hidden=(256, 128), sigma=0.1, bucket=B.BUCKET_MOD, sigmoid=1, zipf=False),
    "base": dict(dtype=B.BF16, d=128, F=16, B=1024, dc=32, hidden=(512, 256), sigma=0.05, bucket=B.BUCKET_HASH, sigmoid=0, zipf=True),
    "wide": dict(dtype=B.BF16, d=256, F=64, B=4096, dc=32, hidden=(1024, 512, 256), sigma=0.05, bucket=B.BUCKET_HASH, sigmoid=0, zipf=True),
}
# The interaction blocks a model is served with: the base model, its long-sequence form with LSH similarities in place of
# the dense attention, both beside each other, and everything on (bridge embeddings too).
BLOCKS = {
    "att": B.BLK_ATT | B.BLK_CROSS,
    "lsh": B.BLK_CROSS | B.BLK_LSH_DIN | B.BLK_SIMTIER,
    "att+lsh": B.BLK_ATT | B.BLK_CROSS | B.BLK_LSH_DIN | B.BLK_SIMTIER,
    "all": B.BLK_ATT | B.BLK_CROSS | B.BLK_BEA | B.BLK_LSH_DIN | B.BLK_SIMTIER,
}
N_BRIDGE, N_TIERS = 8, 8
ITEM_WIDTHS = (4, 2, 1)   # raw item features, hidden width and multi-modal embedding, in multiples of d


def _case(name, call, model, blocks, R, n, L, M, **kw):
    c = dict(name=name, call=call, model=model, blocks=blocks, R=R, n=n, L=L, M=M, mini_batch=0, n_categories=0, mixed=False,
             overlap=0.0)
    c.update(kw)
    return c


def listed():
    return [
        # the fp32 model: one small request
        _case("fp32_request_1000", "score", "small", "att", 1, 1000, 50, 100_000),
        # one mini-batch of the paper's size, the smallest scoring call a serving process makes
        _case("minibatch_1000", "score", "base", "att", 1, 1000, 200, 1_000_000, mini_batch=1000),
        # the headline: one request of 10^4 candidates in ten mini-batches, ids and logits in pinned host memory
        _case("request_1e4_host", "score_host", "base", "att", 1, 10_000, 200, 1_000_000, mini_batch=1000),
        # one request through the model with every block on, a ragged number of candidates
        _case("request_all_blocks", "score", "base", "all", 1, 9_877, 1000, 1_000_000),
        # one request from raw user features: the user-side network and then scoring
        _case("user_and_score", "user+score", "base", "att", 1, 10_000, 1000, 1_000_000),
        # concurrent serving: 64 requests in one call from host memory, 30 % of the ids common to all of them
        _case("concurrent_64_host", "batch_host", "base", "att", 64, 10_000, 1000, 10_000_000, overlap=0.3),
        # long behaviour sequences, dense attention
        _case("long_sequence_att", "batch", "base", "att", 16, 10_000, 10_000, 1_000_000),
        # the same with the LSH similarities in place of the dense attention
        _case("long_sequence_lsh", "batch", "base", "lsh", 16, 10_000, 10_000, 1_000_000),
        # 10^5 behaviours, each candidate against the sub-sequence of its own category
        _case("category_subsequences", "batch", "base", "att+lsh", 4, 10_000, 100_000, 1_000_000, n_categories=100),
        # the wide model, 256 concurrent requests (the largest)
        _case("wide_256_requests", "batch", "wide", "att", 256, 4000, 500, 5_000_000),
        # incremental update of the item table: vectors, bridge weights and signatures of 10^5 items, read back by id
        _case("table_refresh_1e5", "refresh", "base", "all", 1, 100_000, 1, 1_000_000),
        # nearline item side: vectors, bridge weights and signatures of a whole table from raw features, read back
        _case("item_side_compute", "compute", "base", "all", 1, 262_143, 1, 262_143),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["single", "single", "single", "fp32", "user", "batch", "batch", "long", "category", "wide", "refresh", "compute"])
    M = _log(rng, 200_000, 2_000_000)
    if kind == "single":
        return _drawn(rng.choice(["score", "score_host"]), "base", rng.choice(["att", "att", "lsh", "all"]), 1, _log(rng, 200, 20_000),
                      _log(rng, 20, 1000), M, mini_batch=rng.choice([0, 1000]))
    if kind == "fp32":
        return _drawn(rng.choice(["score", "score_host"]), "small", "att", 1, _log(rng, 100, 4000), _log(rng, 10, 200), 100_000)
    if kind == "user":
        return _drawn("user+score", "base", rng.choice(["att", "all"]), 1, _log(rng, 500, 10_000), _log(rng, 50, 10_000), M)
    if kind == "batch":
        return _drawn(rng.choice(["batch", "batch_host"]), "base", rng.choice(["att", "att", "lsh", "all"]), _log(rng, 2, 64), _log(rng, 500, 10_000),
                      _log(rng, 50, 1000), M, mixed=rng.choice([False, True]), overlap=rng.choice([0.0, 0.3]))
    if kind == "long":
        return _drawn("batch", "base", rng.choice(["att", "lsh", "att+lsh"]), _log(rng, 2, 16), _log(rng, 1000, 10_000), _log(rng, 1000, 10_000), M)
    if kind == "category":
        return _drawn("batch", "base", rng.choice(["att", "lsh", "att+lsh"]), rng.randint(1, 4), _log(rng, 2000, 10_000), _log(rng, 10_000, 100_000), M,
                      n_categories=rng.choice([50, 100, 200]))
    if kind == "wide":
        return _drawn(rng.choice(["batch", "batch_host"]), "wide", "att", _log(rng, 4, 256), _log(rng, 500, 4000), _log(rng, 50, 500), M,
                      mixed=rng.choice([False, True]))
    n = _log(rng, 2000, 500_000)
    return _drawn(kind, "base", rng.choice(["att", "all"]), 1, n, 1, n if kind == "compute" else max(M, n))


def _drawn(*a, **kw):
    c = _case("", *a, **kw)
    del c["name"]
    return c


# ---- inputs -----------------------------------------------------------------------------------------------------
class _Inputs:
    """Random inputs on the GPU, from the seed alone."""

    def __init__(self, seed, model):
        self.g = torch.Generator(device="cuda").manual_seed(seed)
        self.m = model
        self.dtype = torch.float32 if model["dtype"] == B.F32 else torch.bfloat16
        self.protos = None

    def normal(self, *shape, sigma=None):
        s = self.m["sigma"] if sigma is None else sigma
        return (torch.randn(*shape, device="cuda", generator=self.g) * s).to(self.dtype)

    def rows(self, n, width):
        """[n, width], drawn in pieces: a table in single precision would need twice its memory on top."""
        out = torch.empty(n, width, dtype=self.dtype, device="cuda")
        for i in range(0, n, 1 << 20):
            out[i:i + (1 << 20)] = self.normal(min(1 << 20, n - i), width)
        return out

    def glorot(self, rows, cols):
        a = math.sqrt(6.0 / (rows + cols))
        return ((torch.rand(rows, cols, device="cuda", generator=self.g) * 2 - 1) * a).to(self.dtype)

    def bias(self, n):
        return torch.randn(n, device="cuda", generator=self.g) * 0.05

    def bridge_weights(self, n):
        e = -torch.log(torch.rand(n, N_BRIDGE, device="cuda", generator=self.g).clamp_min(1e-9))
        return (e / e.sum(1, keepdim=True)).to(self.dtype)

    def signatures(self, n, bits):
        """Rows near one of 16 prototypes with up to half of the bits flipped, packed with the first bit on top."""
        if self.protos is None:
            self.protos = torch.randint(0, 2, (16, bits), device="cuda", generator=self.g, dtype=torch.uint8)
        weights = torch.tensor([128, 64, 32, 16, 8, 4, 2, 1], device="cuda", dtype=torch.uint8)
        out = torch.empty(n, bits // 8, device="cuda", dtype=torch.uint8)
        for i in range(0, n, 1 << 18):
            k = min(1 << 18, n - i)
            which = torch.randint(0, 16, (k,), device="cuda", generator=self.g)
            share = torch.rand(k, 1, device="cuda", generator=self.g) * 0.5
            flip = (torch.rand(k, bits, device="cuda", generator=self.g) < share).to(torch.uint8)
            out[i:i + k] = ((self.protos[which] ^ flip).view(k, bits // 8, 8) * weights).sum(2, dtype=torch.uint8)
        return out

    def ids(self, sizes, M, overlap):
        """Candidate ids of every request, distinct within a request: Zipf (s = 1.1) ranks through a permutation of the
        table, or uniform; a share of every request from one pool common to all."""
        if self.m["zipf"]:
            cdf = torch.cumsum(torch.arange(1, M + 1, device="cuda", dtype=torch.float64) ** -1.1, 0)
            cdf /= cdf[-1].clone()
            perm = torch.randperm(M, device="cuda", generator=self.g)

        def some(k):
            if not self.m["zipf"]:
                return torch.randint(0, M, (k,), device="cuda", generator=self.g)
            u = torch.rand(k, device="cuda", generator=self.g, dtype=torch.float64)
            return perm[torch.searchsorted(cdf, u).clamp_max_(M - 1)]

        def distinct(k, without):
            got = none
            while got.numel() < k:
                got = torch.unique(torch.cat([got, some(4 * k)]))
                got = got[~torch.isin(got, without)]
            return got[torch.randperm(got.numel(), device="cuda", generator=self.g)[:k]]

        none = torch.empty(0, device="cuda", dtype=torch.int64)
        pool = distinct(int(overlap * max(sizes)), none) if overlap else none
        out = []
        for n in sizes:
            shared = pool[:int(overlap * n)]
            ids = torch.cat([shared, distinct(n - shared.numel(), shared)])
            out.append(ids[torch.randperm(n, device="cuda", generator=self.g)].to(torch.int32))
        return torch.cat(out)


def _sizes(case):
    """Candidates of every request: the case's, or spread over [n / 10, n] in a way of the case's own."""
    if not case["mixed"]:
        return [case["n"]] * case["R"]
    g = torch.Generator().manual_seed(case["R"] * case["n"])
    return [int(x) for x in torch.randint(max(1, case["n"] // 10), case["n"] + 1, (case["R"],), generator=g)]


def _config(case, m, blocks, sizes):
    table_only = case["call"] in ("refresh", "compute")
    return B.make_config(
        dtype=m["dtype"], M=case["M"], d=m["d"], L_max=case["L"], hidden=m["hidden"], F=m["F"], B=m["B"], dc=m["dc"],
        bucket_mode=m["bucket"], blocks=blocks, n_bridge=N_BRIDGE, n_tiers=N_TIERS, emit_sigmoid=m["sigmoid"],
        max_user_states=case["R"], mini_batch=case["mini_batch"], n_categories=case["n_categories"],
        max_batch_candidates=128 if table_only else sum(sizes))


def _load_weights(ctx, x, m, blocks):
    width, W, b = ctx.input_width, [], []
    for h in m["hidden"]:
        W.append(x.glorot(h, width))
        b.append(x.bias(h))
        width = h
    d = m["d"]
    user = {"W_profile": x.glorot(d, d), "W_seq": x.glorot(d, d), "W_a": x.glorot(d, d), "W_b": x.glorot(d, d), "b_a": x.bias(d), "b_b": x.bias(d)}
    if blocks & B.BLK_BEA:
        user["bridges"], user["W_f"] = x.normal(N_BRIDGE, d, sigma=1.0), x.glorot(d, d)
    ctx.load_weights({"W": W, "b": b, "w_out": x.glorot(1, width).reshape(-1), "b_out": x.bias(1)}, user)


def _user(case, x, m, blocks, cross):
    """The arguments of user_precompute for one user."""
    d, L = m["d"], case["L"]
    u = {"profile": x.normal(d), "seq": x.normal(L, d), "cross_raw": cross}
    if blocks & B.BLK_BEA:
        u["bea_U" if case["call"] == "user+score" else "bea_V"] = x.normal(64 if case["call"] == "user+score" else N_BRIDGE, d)
    if blocks & B.BLK_LSH_DIN:
        u["seq_sig"] = x.signatures(L, d)
    if case["n_categories"]:   # a few favourite categories and a long tail
        w = 1.0 / (1.0 + torch.randperm(case["n_categories"], device="cuda", generator=x.g))
        u["seq_cat"] = torch.multinomial(w, L, replacement=True, generator=x.g).to(torch.int32)
    return u


def prepare(case, seed):
    m, blocks, call = MODELS[case["model"]], BLOCKS[case["blocks"]], case["call"]
    x = _Inputs(seed, m)
    sizes = _sizes(case)
    d, n, M = m["d"], case["n"], case["M"]
    ctx = B.Aif(_config(case, m, blocks, sizes))
    s = {"ctx": ctx, "call": call}
    if call in ("refresh", "compute"):
        bea, lsh = bool(blocks & B.BLK_BEA), bool(blocks & B.BLK_LSH_DIN)
        if call == "refresh":
            s["ids"] = torch.randperm(M, device="cuda", generator=x.g)[:n].to(torch.int32)
            s["rows"] = x.rows(n, d)
            s["bea_w"] = x.bridge_weights(n) if bea else None
            s["sig"] = x.signatures(n, d) if lsh else None
        else:
            dI, hI, d_mm = (k * d for k in ITEM_WIDTHS)
            s["ids"] = torch.arange(n, device="cuda", dtype=torch.int32)
            s["I_raw"], s["I_id"], s["M_mm"] = x.rows(n, dI), x.normal(n, d, sigma=1.0) if bea else None, x.normal(n, d_mm, sigma=1.0) if lsh else None
            w = {"W_i0": x.glorot(hI, dI), "b_i0": x.bias(hI), "W_i1": x.glorot(d, hI), "b_i1": x.bias(d)}
            if bea:
                w["bridges"] = x.normal(N_BRIDGE, d, sigma=1.0)
            if lsh:
                w["W_hash"] = x.normal(d, d_mm, sigma=1.0)
            ctx.load_item_weights(w)
        s["rows_out"] = torch.empty(n, d, dtype=x.dtype, device="cuda")
        s["bea_out"] = torch.empty(n, N_BRIDGE, dtype=x.dtype, device="cuda") if bea else None
        s["sig_out"] = torch.empty(n, d // 8, dtype=torch.uint8, device="cuda") if lsh else None
        torch.cuda.synchronize()
        return s
    _load_weights(ctx, x, m, blocks)
    ctx.item_nearline_refresh(None, x.rows(M, d), x.bridge_weights(M) if blocks & B.BLK_BEA else None,
                              x.signatures(M, d) if blocks & B.BLK_LSH_DIN else None)
    s["ids"] = x.ids(sizes, M, case["overlap"])
    tables = [x.normal(m["F"], m["B"], m["dc"]) for _ in range(min(case["R"], 16))]
    users = [_user(case, x, m, blocks, tables[r % 16]) for r in range(case["R"])]
    if call == "user+score":
        s["user"] = users[0]
    else:
        s["states"] = [ctx.user_precompute(r, mode=B.USER_PROJECTED, **u) for r, u in enumerate(users)]
    s["offsets"] = [0]
    for k in sizes:
        s["offsets"].append(s["offsets"][-1] + k)
    s["logits"] = torch.empty(sum(sizes), dtype=torch.float32, device="cuda")
    if call.endswith("_host"):
        s["ids"] = s["ids"].cpu().pin_memory()
        s["logits"] = torch.empty(sum(sizes), dtype=torch.float32).pin_memory()
    torch.cuda.synchronize()
    return s


# ---- the pass ---------------------------------------------------------------------------------------------------
def run(s):
    ctx, call = s["ctx"], s["call"]
    if call == "score":
        ctx.score(s["states"][0], s["ids"], s["logits"])
    elif call == "score_host":
        ctx.score_host(s["states"][0], s["ids"], s["logits"])
    elif call == "batch":
        ctx.score_batch(s["states"], s["ids"], s["offsets"], s["logits"])
    elif call == "batch_host":
        ctx.score_batch_host(s["states"], s["ids"], s["offsets"], s["logits"])
    elif call == "user+score":
        # all on one stream, so the slot can be handed back as soon as the scoring call is queued
        state = ctx.user_precompute(1, mode=B.USER_RAW, **s["user"])
        ctx.score(state, s["ids"], s["logits"])
        state.release()
    else:
        if call == "refresh":
            ctx.item_nearline_refresh(s["ids"], s["rows"], s["bea_w"], s["sig"])
        else:
            ctx.item_nearline_compute(None, s["I_raw"], s["I_id"], s["M_mm"])
        ctx.gather_rows(s["ids"], s["rows_out"])
        if s["bea_out"] is not None:
            ctx.gather_sidecars(s["ids"], s["bea_out"], s["sig_out"])
        return {"rows": s["rows_out"], "bea_w": s["bea_out"], "sig": s["sig_out"]}
    return s["logits"]


# ---- what a pass cannot do without ------------------------------------------------------------------------------
def work(case):
    m, blocks = MODELS[case["model"]], BLOCKS[case["blocks"]]
    el, d, n, R, L = (4 if m["dtype"] == B.F32 else 2), m["d"], case["n"], case["R"], case["L"]
    side = (N_BRIDGE * el if blocks & B.BLK_BEA else 0) + (d // 8 if blocks & B.BLK_LSH_DIN else 0)
    if case["call"] == "refresh":      # ids and rows in, table rows written; ids again, table rows read, rows out
        return {"bytes": n * (4 * (d * el + side) + 8), "flops": 0}
    if case["call"] == "compute":
        dI, hI, d_mm = (k * d for k in ITEM_WIDTHS)
        inputs = dI + (d if blocks & B.BLK_BEA else 0) + (d_mm if blocks & B.BLK_LSH_DIN else 0)
        flops = 2 * (dI * hI + hI * d) + (2 * N_BRIDGE * d if blocks & B.BLK_BEA else 0) + (2 * d_mm * d if blocks & B.BLK_LSH_DIN else 0)
        return {"bytes": n * (inputs * el + 3 * (d * el + side) + 4), "flops": n * flops}
    total = sum(_sizes(case))
    keys = L / case["n_categories"] if case["n_categories"] else L
    width = d + m["F"] * m["dc"] + N_TIERS * bool(blocks & B.BLK_SIMTIER)
    flops = 0.0
    for blk, per in ((B.BLK_ATT, 4 * keys * d), (B.BLK_LSH_DIN, 2 * keys * d), (B.BLK_BEA, 2 * N_BRIDGE * d)):
        if blocks & blk:
            flops, width = flops + per, width + d
    weights = 0
    for h in m["hidden"]:
        flops, weights, width = flops + 2 * width * h, weights + width * h, h
    flops += 2 * width
    per_user = L * (d * el + (d // 8 if blocks & B.BLK_LSH_DIN else 0)) + m["F"] * min(m["B"], total / R) * m["dc"] * el
    user_flops = 0
    if case["call"] == "user+score":   # eqs. 1-3: projection, self-attention, FFN hidden layer, profile attention; p_u
        user_flops = 2 * L * d * d + 4 * L * L * d + 2 * L * d * d + 4 * L * d + 2 * d * (3 * d + m["hidden"][0])
        per_user += m["F"] * m["B"] * m["dc"] * el * 2   # the cross pre-cache is copied
    return {"bytes": total * (d * el + side + 8) + R * per_user + weights * el, "flops": total * flops + R * user_flops}


def tolerance(case):
    """fp32: sums of a few hundred terms.  bf16: activations and attention rows are rounded to bf16 between the layers
    (2^-9 each).  A signature bit is the sign of a bf16 projection accumulated in fp32: one within rounding of zero may
    fall either way, fewer than 1 byte in 500."""
    if case["call"] == "refresh":
        return "exact"
    if MODELS[case["model"]]["dtype"] == B.F32:
        return {"rel": 1e-5}
    return {"rel": 1e-2, "differ": 2e-3} if case["call"] == "compute" else {"rel": 1e-2}
