"""LSH-DIN through the requests' own sums and SimTier counted by itself, against the CPU oracle: sequences at the edges of
their key blocks and units, numbers of tiers whose boundaries are no binary fractions, both widths, and scaled outputs off."""
import numpy as np
import pytest
import torch

from paper_2511_12934_b200 import binding as B
from paper_2511_12934_b200 import build as libbuild
from paper_2511_12934_b200 import serving, synth
from tests import helpers

pytestmark = pytest.mark.gpu
LSH = synth.BLK_LSH_DIN | synth.BLK_SIMTIER


@pytest.fixture(scope="module", autouse=True)
def _built():
    libbuild.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    B.load_library()


def _run(base, blocks, Ls, sizes, one_by_one=(), more=None, route=(), **kw):
    """more: (request, candidates that it has besides, which make the launch a large one); route: kernels that the launch has to take."""
    extra = more[1] if more else 0
    wl = helpers.MINI[base].with_(name=f"lsh_sums_{base}_{blocks}", R=len(Ls), N=max(sizes), L=max(Ls), mini_batch=0, blocks=blocks, **kw)
    weights, table = synth.make_weights(wl, zero_bias=False), None
    table = synth.make_item_table(wl)
    srv = serving.Server(wl, weights, table, path=B.PATH_TENSOR, max_batch_candidates=sum(sizes) + extra)
    oracle = helpers.make_oracle(wl, weights, M=table["E"].shape[0])
    sampler = synth.IdSampler(wl)
    states, ids, want = [], [], []
    for r, (L, n) in enumerate(zip(Ls, sizes)):
        rq = synth.make_request(wl, r, L=L)
        states.append(srv.precompute(r, srv.upload_request(rq, B.USER_PROJECTED)))
        ids.append(sampler.request_ids(r, n))
        want.append(oracle.score(table, helpers.projected_request(wl, rq), ids[-1]))
    whole = [np.concatenate([i, np.resize(ids[0], extra)]) if more and r == more[0] else i for r, i in enumerate(ids)]
    srv.ctx.set_kernel_timing(True)
    outs = [o[:len(i)] for o, i in zip(srv.score_many(states, whole), ids)]
    assert set(route) <= set(srv.ctx.get_kernel_timing())
    srv.ctx.set_kernel_timing(False)
    for r in one_by_one:
        outs.append(srv.score_ids(states[r], ids[r])), want.append(want[r])
    for r, (o, w) in enumerate(zip(outs, want)):
        err = float(np.abs(o.astype(np.float64) - w).max())
        assert err <= 2e-3, (r, err)
    assert srv.ctx.poll_status() == 0
    srv.close()


@pytest.mark.parametrize("n_tiers", [1, 2, 3, 5, 6, 7, 8, 9])
def test_numbers_of_tiers(n_tiers):
    """One to eight tiers by the bit-sliced counters (nine: the other kernel), with and without LSH-DIN beside them."""
    _run("c2", synth.BLK_CROSS | LSH, [700, 513], [200, 129], n_tiers=n_tiers)
    _run("c2", synth.BLK_CROSS | synth.BLK_SIMTIER, [700, 130], [130, 77], n_tiers=n_tiers)


# One long sequence with many candidates makes the launch a large one, which is what takes LSH-DIN to the sums; the others are at the edges.
@pytest.mark.parametrize("base,blocks", [("c2", synth.BLK_CROSS | LSH), ("c2", helpers.ALL_BLOCKS), ("c2", synth.BLK_CROSS | synth.BLK_LSH_DIN),
                                         ("c5", synth.BLK_CROSS | LSH), ("c5", synth.BLK_ATT | synth.BLK_CROSS | LSH)])
def test_sequences_at_the_edges_of_blocks_and_units(base, blocks):
    """Key blocks and units of 128 (64 for the pieces at d = 256), up to eight CTAs per request: lengths on either side of each, requests of
    one candidate and of a whole number of tiles, scored together and, a few, alone (the pass over the pairs)."""
    Ls = [1, 63, 65, 127, 128, 129, 255, 256, 257, 385, 640, 1025, 40_001]
    sizes = [1, 127, 128, 129, 33, 300, 64, 31, 256, 1, 130, 700, 2]
    _run(base, blocks, Ls, sizes, one_by_one=(9, 10, 11), more=(12, 2500), route=("lsh_sums", "lsh_rows"))


def test_pieces_of_long_sequences():
    """Fewer tiles than SMs: SimTier's counts in pieces of the keys; one tile over a sequence that a counter's lower digits do not hold."""
    _run("c2", synth.BLK_CROSS | LSH, [9001, 4096], [5300, 128], one_by_one=(1,), route=("lsh_sums", "simtier"))
    _run("c2", synth.BLK_CROSS | synth.BLK_SIMTIER, [70_000], [3])
    _run("c5", synth.BLK_CROSS | synth.BLK_SIMTIER, [3001], [100])


@pytest.mark.parametrize("base,L", [("c2", 2600), ("c5", 4200)])
def test_more_requests_than_sms(base, L):
    """One CTA per request and column half."""
    n = 160
    _run(base, synth.BLK_CROSS | LSH, [L] + [40 + r for r in range(n - 1)], [3 + r % 5 for r in range(n)], one_by_one=(0,), more=(0, 26_000), route=("lsh_sums", "simtier"))


# ---- the columns themselves -------------------------------------------------------------------------------------------
# One hidden layer of which two units pass sum_c r_c x_c on, its positive and its negative part: the logit is that sum over the LSH-DIN
# or SimTier columns as the layer reads them (bf16).  Rounding to bf16's eight significant bits costs at most 2^-8 of each column and of the
# sum, which is the tolerance (and 1 % of it for fp32 and second-order terms); a scoring network of random weights hides most of what can be wrong in
# a few of its inputs.
BF16 = 2.0 ** -8


def _columns(wl, blk):
    at = 2 * wl.d + (wl.d if wl.blocks & synth.BLK_ATT else 0) + (wl.F * wl.dc if wl.blocks & synth.BLK_CROSS else 0)
    at += wl.d if wl.blocks & synth.BLK_BEA else 0
    if blk == synth.BLK_LSH_DIN:
        return at, wl.d
    return at + (wl.d if wl.blocks & synth.BLK_LSH_DIN else 0), wl.n_tiers


def _probe(wl, blk, which):
    """Row of factors over the input columns: random signs over the block's (different ones per `which`); first, over tiers, a ramp about
    zero, which every pair that is in the next tier moves by two."""
    at, n = _columns(wl, blk)
    r = np.zeros(wl.input_width(), np.float32)
    r[at:at + n] = np.random.default_rng(100 * n + which).choice([-1.0, 1.0], n)
    if blk == synth.BLK_SIMTIER and which == 0 and n > 1:
        r[at:at + n] = 2.0 * np.arange(n) - (n - 1)
    return r


def _load(ctx, r):
    W = torch.zeros(64, r.size, dtype=torch.bfloat16, device="cuda")
    W[0], W[1] = torch.from_numpy(r).cuda(), -torch.from_numpy(r).cuda()
    w_out = torch.zeros(64, dtype=torch.bfloat16, device="cuda")
    w_out[0], w_out[1] = 1, -1
    ctx.load_weights({"W": [W], "b": [torch.zeros(64, device="cuda")], "w_out": w_out, "b_out": torch.zeros(1, device="cuda")})


def _sums(x, r):
    """What the logit has to be and how far off it may be."""
    a = x @ r.astype(np.float64)
    return a, 1.01 * BF16 * (np.abs(x) @ np.abs(r).astype(np.float64) + np.abs(a)) + 1e-6


def _without_block(rq, b):
    """The request with the rows of key block b (of 128) at zero."""
    out = dict(rq, S=rq["S"].copy())
    out["S"][128 * b:128 * b + 128] = 0.0
    return out


def _tiers_shifted(wl, table, rq, ids):
    """SimTier columns with every tier's edge one match lower."""
    bits = lambda a: np.unpackbits(a, axis=1).astype(np.float32) * 2 - 1
    m = ((bits(table["sig"][ids]) @ bits(rq["sig_seq"]).T + wl.d) / 2).astype(np.int64)
    t = np.minimum((m + 1) * wl.n_tiers // wl.d, wl.n_tiers - 1)
    x = np.stack([(t == k).sum(1) for k in range(wl.n_tiers)], 1).astype(np.float64)
    return x / (m.shape[1] if wl.simtier_norm == synth.NORM_MEAN else 1)


class Columns:
    """A context over a workload's requests whose LSH columns are read by probes.  more: as for _run."""

    def __init__(self, base, blocks, Ls, sizes, M=5000, change=None, more=None, **kw):
        self.wl = wl = helpers.MINI[base].with_(name=f"lsh_cols_{base}", R=len(Ls), N=max(sizes), M=M, L=max(Ls), mini_batch=0, blocks=blocks,
                                                hidden=(64,), **{"n_cross_tables": 2, **kw})
        weights = synth.make_weights(wl)
        self.table = synth.make_item_table(wl)
        self.rqs = [synth.make_request(wl, r, L=L) for r, L in enumerate(Ls)]
        sampler = synth.IdSampler(wl)
        self.ids = [sampler.request_ids(r, n) for r, n in enumerate(sizes)]
        if change:
            change(self)
        self.more = more or (0, 0)
        self.srv = serving.Server(wl, weights, self.table, path=B.PATH_TENSOR, max_batch_candidates=sum(sizes) + self.more[1])
        self.up = [self.srv.upload_request(rq, B.USER_PROJECTED) for rq in self.rqs]
        oracle = helpers.make_oracle(wl, weights, M=M)
        self.oracle = lambda r, rq=None: oracle.score(self.table, rq or helpers.projected_request(wl, self.rqs[r]), self.ids[r], return_inputs=True)[1]
        self.x = [self.oracle(r) for r in range(len(Ls))]

    def score(self, states):
        whole = [np.concatenate([i, np.resize(self.ids[0], self.more[1])]) if k == self.more[0] else i for k, i in enumerate(self.ids)]
        return [o[:len(i)] for o, i in zip(self.srv.score_many(states, whole), self.ids)]

    def read(self, r, alone=False):
        """Logits of every request under the probe r, and the kernels of the (last) call."""
        _load(self.srv.ctx, r)
        for s in [self.srv.precompute(0, self.up[int(np.argmax([len(rq["S"]) for rq in self.rqs]))]) for _ in self.up]:
            s.release()   # (every slot has held the longest sequence before)
        st = [self.srv.precompute(k, u) for k, u in enumerate(self.up)]
        self.srv.ctx.set_kernel_timing(True)
        outs = [self.srv.score_ids(s, i) for s, i in zip(st, self.ids)] if alone else self.score(st)
        names = set(self.srv.ctx.get_kernel_timing())
        self.srv.ctx.set_kernel_timing(False)
        for s in st:
            s.release()
        return outs, names

    def check(self, blk, route, probes=(0, 1, 2), alone=False, sharp=(), skip=()):
        """Every request's block against the oracle, by the kernels `route`; for the requests `sharp` the oracle's values for a wrong answer (a key
        block left out: the last where it holds eight keys of a thousand, else the first, and three of a long sequence's; tiers one match off) lie
        outside the tolerance."""
        visible = {}
        for which in probes:
            r = _probe(self.wl, blk, which)
            outs, names = self.read(r, alone=alone)
            assert route <= names, names
            for k, (o, x) in enumerate(zip(outs, self.x)):
                if k in skip:
                    continue
                want, tol = _sums(x, r)
                err = np.abs(o.astype(np.float64) - want)
                assert (err <= tol).all(), (k, which, float((err / tol).max()))
                if blk == synth.BLK_SIMTIER and self.wl.simtier_norm == synth.NORM_NONE and len(self.rqs[k]["S"]) <= 256 // np.abs(r).max():
                    assert np.array_equal(o, want), (k, which)   # counts that bf16 holds
                if k not in sharp:
                    continue
                if blk == synth.BLK_SIMTIER:
                    at, n = _columns(self.wl, blk)
                    wrong = {k: _tiers_shifted(self.wl, self.table, self.rqs[k], self.ids[k]) @ r[at:at + n].astype(np.float64)}
                else:
                    L, rq = len(self.rqs[k]["S"]), helpers.projected_request(self.wl, self.rqs[k])
                    nb = (L + 127) // 128
                    gone = [0, nb // 2, nb - 1] if L > 10_000 else [nb - 1 if 125 * ((L - 1) % 128 + 1) >= L else 0]
                    wrong = {(k, b): _sums(self.oracle(k, _without_block(rq, b)), r)[0] for b in gone}
                for what, w in wrong.items():
                    visible.setdefault(what, []).append((np.abs(w - want) > 2 * tol).any())
        assert all(any(v) for v in visible.values()), visible
        return self


SUMS, TIERS = {"lsh_sums", "lsh_rows"}, {"simtier"}


@pytest.mark.parametrize("base,blocks", [("c2", LSH), ("c2", helpers.ALL_BLOCKS), ("c2", synth.BLK_LSH_DIN), ("c5", LSH), ("c5", synth.BLK_ATT | LSH)])
def test_columns_at_the_edges_of_blocks_and_units(base, blocks):
    """The launch of many key blocks above, its columns read by probes: a dropped key block shows in every request of more than one; so does a
    tier's edge that is off by one match.  Of the 313 blocks of the longest (over eight CTAs) the first, the middle and the last have
    rows four times as large, so that one of them is more than the columns' rounding."""
    Ls = [1, 63, 65, 127, 128, 129, 255, 256, 257, 385, 640, 1025, 40_001]
    sizes = [1, 127, 128, 129, 33, 300, 64, 31, 256, 40, 130, 700, 24]
    def emphasise(c):
        S = c.rqs[12]["S"]
        for b in (0, 156, 312):
            S[128 * b:128 * b + 128] = synth.to_bf16_bits(4.0 * synth.bf16_bits_to_f32(S[128 * b:128 * b + 128]))
    c = Columns(base, blocks, Ls, sizes, change=emphasise, more=(12, 2500))
    c.check(synth.BLK_LSH_DIN, SUMS, sharp=(5, 6, 7, 8, 9, 10, 11, 12))
    if blocks & synth.BLK_SIMTIER:
        c.check(synth.BLK_SIMTIER, SUMS | TIERS, sharp=(3, 4, 5, 6, 7, 8, 9, 10, 11, 12))
    c.srv.close()


def _same_and_opposite(c):
    """Request 2's keys carry the signature of its first candidate, then the complement: d' matches and none."""
    sig = c.table["sig"][c.ids[2][0]]
    c.rqs[2]["sig_seq"][:130], c.rqs[2]["sig_seq"][130:] = sig, ~sig


@pytest.mark.parametrize("base", ["c2", "c5"])
@pytest.mark.parametrize("n_tiers", [1, 2, 3, 4, 5, 6, 7, 8])
def test_tier_counts_column_by_column(base, n_tiers):
    """Every number of tiers that the bit-sliced counters take, beside the sums and by themselves, with counts at both ends of their range."""
    Ls, sizes, sharp = [700, 513, 256, 9001], [200, 129, 60, 40], (0, 1, 3) if n_tiers > 1 else ()
    c = Columns(base, LSH, Ls, sizes, change=_same_and_opposite, more=(3, 9000), n_tiers=n_tiers)
    c.check(synth.BLK_SIMTIER, SUMS | TIERS, sharp=sharp).check(synth.BLK_LSH_DIN, SUMS, probes=(0,))
    c.srv.close()
    c = Columns(base, synth.BLK_SIMTIER, Ls, sizes, change=_same_and_opposite, n_tiers=n_tiers)
    c.check(synth.BLK_SIMTIER, {"lsh"}, sharp=sharp).check(synth.BLK_SIMTIER, {"lsh"}, alone=True, probes=(0,))
    c.srv.close()


@pytest.mark.parametrize("base", ["c2", "c5"])
def test_sums_and_counts_that_are_not_divided_by_the_length(base):
    """Eqs. 8 and 9 as printed: sums of up to 9001 rows, counts that bf16 holds exactly where the sequence is short."""
    c = Columns(base, LSH, [36, 129, 256, 9001], [300, 129, 60, 40], change=_same_and_opposite, more=(3, 9000), lsh_din_norm=synth.NORM_NONE,
                simtier_norm=synth.NORM_NONE)
    c.check(synth.BLK_SIMTIER, SUMS | TIERS, sharp=(0, 1, 2, 3)).check(synth.BLK_LSH_DIN, SUMS, sharp=(1, 2, 3))
    c.srv.close()


def test_counts_of_keys_by_category():
    """SimTier alone over the tables of jobs: groups of many key blocks in pieces, groups of a few keys, categories without any."""
    c = Columns("c2", synth.BLK_SIMTIER, [30_000, 500, 20], [900, 300, 40], n_categories=13)
    c.check(synth.BLK_SIMTIER, {"lsh", "group"})
    c.srv.close()
    c = Columns("c5", synth.BLK_SIMTIER, [9000, 300], [500, 200], n_categories=5, n_tiers=7)
    c.check(synth.BLK_SIMTIER, {"lsh", "group"})
    c.srv.close()


def test_counters_that_one_piece_fills():
    """As many tiles as SMs, so that a CTA takes all of a tile's keys: 10^4 of them run over the lower binary digits of a counter (every key in one tier),
    1 060 000 over what both halves hold, after which they are emptied on the way."""
    tiles = 148 * 128
    def nearly_all_opposite(c):
        c.rqs[0]["sig_seq"][100:] = ~c.table["sig"][c.ids[0][0]]
    c = Columns("c2", synth.BLK_SIMTIER, [10_100], [40], change=nearly_all_opposite, more=(0, tiles - 40))
    assert c.x[0][0, _columns(c.wl, synth.BLK_SIMTIER)[0]] > 0.98
    c.check(synth.BLK_SIMTIER, {"lsh"}, sharp=(0,))
    c.srv.close()

    L, d, N = 1_060_000, 128, 8
    g = torch.Generator(device="cuda").manual_seed(5)
    ctx = B.Aif(B.make_config(dtype=B.BF16, M=1000, d=d, L_max=L, hidden=(64,), blocks=synth.BLK_SIMTIER, n_tiers=N, lsh_bits=d, max_user_states=1,
                              max_batch_candidates=tiles, simtier_norm=synth.NORM_MEAN))
    item = torch.randint(0, 256, (1000, d // 8), device="cuda", generator=g, dtype=torch.uint8)
    keys = torch.randint(0, 256, (L, d // 8), device="cuda", generator=g, dtype=torch.uint8)
    keys[5000:900_000] = ~item[0]   # candidate 0: nine tenths of the keys in the first tier
    ctx.item_nearline_refresh(None, torch.zeros(1000, d, dtype=torch.bfloat16, device="cuda"), None, item)
    r = np.zeros(ctx.input_width, np.float32)
    r[2 * d:2 * d + N] = 2.0 * np.arange(N) - (N - 1)
    _load(ctx, r)
    st = ctx.user_precompute(0, mode=B.USER_PROJECTED, profile=torch.zeros(d, dtype=torch.bfloat16, device="cuda"),
                             seq=torch.zeros(L, d, dtype=torch.bfloat16, device="cuda"), seq_sig=keys)
    ids = (torch.arange(tiles, device="cuda") % 1000).to(torch.int32)
    out = torch.empty(tiles, device="cuda")
    ctx.score(st, ids, out)
    got = out[:16].cpu().numpy()
    bits = lambda a: np.unpackbits(a.cpu().numpy(), axis=1).astype(np.float32) * 2 - 1
    m = ((bits(item[:16]) @ bits(keys).T + d) / 2).astype(np.int64)
    t = np.minimum(m * N // d, N - 1)
    want, tol = _sums(np.stack([(t == k).sum(1) for k in range(N)], 1) / L, r[2 * d:2 * d + N])
    assert (np.abs(got - want) <= tol).all(), np.abs(got - want) / tol
    # a counter that had lost what it was emptied of (65 280 keys of a warp) would be off by more
    assert (16 * 65_280 / 4 / L * 2 > 2 * tol[0]) and ctx.poll_status() == 0
    ctx.close()


def test_a_launch_of_more_requests_than_a_round_of_sums():
    """300 requests, of none to a few hundred candidates, go in a round of 256 and one of the rest; one state serves two of them."""
    n = 300
    sizes = [(3 + 7 * k % 260) if k % 11 else 0 for k in range(n)]
    sizes[0], sizes[255], sizes[256], sizes[299] = 5, 0, 130, 129
    c = Columns("c2", synth.BLK_LSH_DIN, [9000] + [40 + k for k in range(n - 1)], [max(1, k) for k in sizes], more=(0, 20_000), n_cross_tables=1)
    c.ids = [i[:k] for i, k in zip(c.ids, sizes)]
    r = _probe(c.wl, synth.BLK_LSH_DIN, 0)
    _load(c.srv.ctx, r)
    st = [c.srv.precompute(k, u) for k, u in enumerate(c.up)]
    st[257], c.ids[257], c.x[257] = st[256], c.ids[256], c.x[256]   # (and a state twice)
    c.srv.ctx.set_kernel_timing(True)
    outs = c.score(st)
    assert SUMS <= set(c.srv.ctx.get_kernel_timing())
    for k, o in enumerate(outs):
        want, tol = _sums(c.x[k][:len(o)], r)
        assert (np.abs(o - want) <= tol).all(), k
    c.srv.close()


def test_room_for_the_sums_does_not_grow_with_the_states_of_a_context():
    """Sums are a request's of a launch, not a state's: 2000 states take the room of a round of requests."""
    def held(blocks):
        ctx = B.Aif(B.make_config(dtype=B.BF16, M=1000, d=128, L_max=384, hidden=(64,), blocks=blocks, n_tiers=8, lsh_bits=128, max_user_states=2000,
                                  max_batch_candidates=4096))
        n = ctx.get_stats().device_bytes
        ctx.close()
        return n
    assert held(LSH) - held(synth.BLK_SIMTIER) < 50 << 20


@pytest.mark.parametrize("base,blocks,R,n,L,sums", [
    ("c2", LSH, 8, 1000, 6000, True), ("c2", LSH, 148, 128, 4000, False), ("c2", LSH, 300, 60, 1500, False),
    ("c2", synth.BLK_LSH_DIN, 32, 256, 7000, True), ("c2", synth.BLK_LSH_DIN, 148, 128, 4000, False),
    ("c5", LSH, 4, 4000, 5000, True), ("c5", LSH, 32, 256, 10_000, False), ("c5", synth.BLK_LSH_DIN, 148, 128, 4200, False)])
def test_sums_are_for_requests_of_many_candidates(base, blocks, R, n, L, sums):
    """The sums are a pass over every request's keys: requests of a tile or two go by the pass over the pairs, which is one as well and needs no other
    launch, however many they are."""
    wl = helpers.MINI[base].with_(name="lsh_route", R=R, N=n, M=5000, L=L, mini_batch=0, blocks=blocks, hidden=(64,))
    srv = serving.Server(wl, synth.make_weights(wl), synth.make_item_table(wl), path=B.PATH_TENSOR)
    up = srv.upload_request(synth.make_request(wl, 0), B.USER_PROJECTED)
    states = [srv.precompute(r, up) for r in range(R)]
    srv.ctx.set_kernel_timing(True)
    srv.score_many(states, [synth.IdSampler(wl).request_ids(0)] * R)
    names = set(srv.ctx.get_kernel_timing())
    assert (SUMS <= names) == sums and ("lsh" in names) == (not sums)
    srv.close()


def test_marks_of_a_call_with_four_layers_and_every_block():
    """Ten kernels and eight entries: the LSH blocks' are reported as one, the others by themselves, nothing is lost."""
    wl = helpers.MINI["c2"].with_(name="lsh_marks", R=1, N=6000, L=9000, mini_batch=0, blocks=helpers.ALL_BLOCKS, hidden=(512, 256, 128, 64))
    srv = serving.Server(wl, synth.make_weights(wl), synth.make_item_table(wl), path=B.PATH_TENSOR)
    st = srv.precompute(0, srv.upload_request(synth.make_request(wl, 0), B.USER_PROJECTED))
    ids = synth.IdSampler(wl).request_ids(0)
    srv.ctx.set_kernel_timing(True)
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    srv.score_ids(st, ids)
    a.record()
    srv.score_ids(st, ids)
    b.record()
    torch.cuda.synchronize()
    marks = srv.ctx.get_kernel_timing()
    assert set(marks) == {"lsh", "attention", "bea", "buckets", "layer1", "layer2", "layer3", "layer4"}
    assert 0.0 < sum(marks.values()) <= a.elapsed_time(b)
    # what the scores hang on most, the pass over the pairs, is under "lsh"
    assert marks["lsh"] > max(marks[k] for k in ("layer2", "layer3", "layer4"))
    srv.close()


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("base", ["c2", "c5"])
@pytest.mark.parametrize("long", [False, True])
def test_rows_that_are_not_finite(base, value, long):
    """A sequence row with one infinite or missing value, by the pass over the pairs and by the sums: the value's column takes its sign (or is
    missing) for every candidate, and is missing where an infinity meets no match at all (0 x inf); a probe of that column alone
    would be no number if any other column were not finite; and the requests beside it are as ever."""
    col, row = 5, 17

    def poison(c):
        bits = np.array([value], np.float32).view(np.uint32)[0] >> 16
        c.rqs[0]["S"][row, col] = bits
        c.table["sig"][c.ids[0][3]] = ~c.rqs[0]["sig_seq"][row]   # candidate 3 shares no bit with the row
    c = Columns(base, LSH, [300, 200] + [40_001] * long, [2000, 300] + [30] * long, change=poison, more=(2, 2500) if long else None)
    at = _columns(c.wl, synth.BLK_LSH_DIN)[0]
    r = np.zeros(c.wl.input_width(), np.float32)
    r[at + col] = 1.0
    outs, names = c.read(r)
    assert (SUMS <= names) == long
    x = c.x[0][:, at + col]
    assert np.isnan(x[3]) and (np.isnan(x).all() if np.isnan(value) else (np.delete(x, 3) == value).all())
    assert np.isfinite(np.delete(c.x[0], at + col, axis=1)).all()
    assert np.array_equal(outs[0], np.where(np.isnan(x), 0.0, x))   # (both units of a missing value are switched off)
    for blk in (synth.BLK_LSH_DIN, synth.BLK_SIMTIER):
        c.check(blk, SUMS | TIERS if long else {"lsh"}, probes=(0,), skip=(0,))
    c.srv.close()
