"""The kernels' own edges: sizes around the tiles, steps and unit widths at which a launch changes what it does, each against
the CPU oracle or a plain numpy statement of the same operation."""
import numpy as np
import pytest
import torch

from oracle import aif_oracle as orc
from paper_2511_12934_b200 import binding as B
from paper_2511_12934_b200 import build as libbuild
from paper_2511_12934_b200 import serving, synth
from tests import helpers

pytestmark = pytest.mark.gpu

TOL = 2e-3


@pytest.fixture(scope="module", autouse=True)
def _built():
    libbuild.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    B.load_library()


def _check(got, want, tol=TOL):
    assert np.array_equal(np.isnan(got), np.isnan(want))
    ok = ~np.isnan(want)
    err = np.abs(got[ok].astype(np.float64) - want[ok]).max() if ok.any() else 0.0
    assert err <= tol, f"max |delta| = {err:.3e} > {tol}"


def _bridge_weights_by_scoring(ctx, n):
    """The bridge weights of items 0 .. n - 1 as the scoring kernels read them, exactly: V's rows are unit vectors, so a column of the
    bridge embedding is one weight; the only layer passes it on, its positive and its negative part in units of their own.  (Rows of
    an odd number of bf16 weights cannot be gathered.)"""
    c, nb = ctx.cfg, ctx.cfg.n_bridge
    H, width, col = c.hidden[0], ctx.input_width, 2 * c.d
    assert H >= 32 and not c.blocks & (B.BLK_ATT | B.BLK_CROSS)
    W1 = torch.zeros(H, width, dtype=ctx.torch_dtype, device="cuda")
    for k in range(nb):
        W1[k, col + k], W1[16 + k, col + k] = 1, -1
    zeros = torch.zeros(c.d, dtype=ctx.torch_dtype, device="cuda")
    V = torch.eye(nb, c.d, dtype=ctx.torch_dtype, device="cuda")
    sig = torch.zeros(1, c.lsh_bits // 8, dtype=torch.uint8, device="cuda") if c.blocks & B.BLK_LSH_DIN else None
    ids = torch.arange(n, dtype=torch.int32, device="cuda")
    out = torch.empty(nb, n, dtype=torch.float32, device="cuda")
    for k in range(nb):
        w_out = torch.zeros(H, dtype=ctx.torch_dtype, device="cuda")
        w_out[k], w_out[16 + k] = 1, -1
        ctx.load_weights({"W": [W1], "b": [torch.zeros(H, device="cuda")], "w_out": w_out, "b_out": torch.zeros(1, device="cuda")})
        st = ctx.user_precompute(k, mode=B.USER_PROJECTED, profile=zeros, seq=zeros.view(1, -1), bea_V=V, seq_sig=sig)
        ctx.score(st, ids, out[k])
        torch.cuda.synchronize()
        st.release()
    return out.t().cpu()


@pytest.mark.parametrize("dtype,d,nb,bits", [("bf16", 128, 8, 128), ("bf16", 64, 3, 64), ("bf16", 96, 16, 32), ("bf16", 256, 5, 256),
                                             ("f32", 64, 8, 96), ("f32", 160, 1, 160), ("f32", 256, 16, 256)])
def test_refresh_and_gathers_at_every_row_width_and_unit(dtype, d, nb, bits):
    """Incremental refresh and both gathers: row widths that fill a group of lanes, do not, or need two rounds of it; sidecar
    rows moved 16, 8, 4 and 2 bytes at a time (also because the caller's sidecar starts off a 16-byte boundary); counts
    around a warp's step; ids outside the table."""
    dt, M = (B.F32 if dtype == "f32" else B.BF16), 3000
    ctx = B.Aif(B.make_config(dtype=dt, M=M, d=d, L_max=8, hidden=(64,), blocks=B.BLK_BEA | B.BLK_LSH_DIN, n_bridge=nb, lsh_bits=bits,
                              max_batch_candidates=M))
    g = torch.Generator().manual_seed(d + nb)
    E, W, S = torch.zeros(M, d, dtype=ctx.torch_dtype), torch.zeros(M, nb, dtype=ctx.torch_dtype), torch.zeros(M, bits // 8, dtype=torch.uint8)
    for n in (1, 15, 16, 17, 63, 65, 1000):
        ids = torch.randperm(M, generator=g)[:n].to(torch.int32)
        rows = torch.randn(n, d, generator=g).to(ctx.torch_dtype)
        bw = torch.randn(n + 1, nb, generator=g).to(ctx.torch_dtype)
        sg = torch.randint(0, 256, (n + 1, bits // 8), generator=g, dtype=torch.uint8)
        if n > 16:
            ids[3], ids[n - 1] = -1, M
        good = (ids >= 0) & (ids < M)
        k = n % 2    # every other count: sidecars that start one row into their buffer
        ctx.item_nearline_refresh(ids.cuda(), rows.cuda(), bw.cuda()[k:k + n], sg.cuda()[k:k + n])
        E[ids[good].long()], W[ids[good].long()], S[ids[good].long()] = rows[good], bw[k:k + n][good], sg[k:k + n][good]
        assert ctx.poll_status() == (0 if good.all() else B.STATUS_BAD_ID)
    for n in (1, 31, 32, 33, M):
        ids = torch.randperm(M, generator=g)[:n].to(torch.int32)
        out = torch.empty(n, d, dtype=ctx.torch_dtype, device="cuda")
        ow = torch.empty(n + 1, nb, dtype=ctx.torch_dtype, device="cuda")
        os_ = torch.empty(n + 1, bits // 8, dtype=torch.uint8, device="cuda")
        ctx.gather_rows(ids.cuda(), out)
        if nb * out.element_size() % 4 == 0:
            ctx.gather_sidecars(ids.cuda(), ow[1:] if ow[1:].data_ptr() % 4 == 0 else ow[:n], os_[1:])
            got = ow[1:] if ow[1:].data_ptr() % 4 == 0 else ow[:n]
            assert torch.equal(got.cpu(), W[ids.long()])
        else:
            ctx.gather_sidecars(ids.cuda(), None, os_[1:])
        assert torch.equal(out.cpu(), E[ids.long()]) and torch.equal(os_[1:].cpu(), S[ids.long()])
    assert torch.equal(_bridge_weights_by_scoring(ctx, M), W.float())
    assert ctx.poll_status() == 0
    ctx.close()


@pytest.mark.parametrize("d", [64, 128, 256])
@pytest.mark.parametrize("nb", [1, 7, 8, 9, 16])
def test_bridge_weights_of_the_nearline_call(d, nb):
    """Algorithm 1 step 3 on the matrix instructions: one and two slices of eight bridges, odd numbers of them, item counts
    around the 16 of a warp.  A weight is at most 1 and is rounded to bf16 once (2^-9)."""
    M = 700
    ctx = B.Aif(B.make_config(dtype=B.BF16, M=M, d=d, L_max=8, hidden=(64,), blocks=B.BLK_BEA, n_bridge=nb, max_batch_candidates=M))
    g = torch.Generator(device="cuda").manual_seed(nb)

    def draw(*shape):
        return torch.randn(*shape, generator=g, device="cuda").to(torch.bfloat16)

    w = {"W_i0": draw(64, 64) * 0.1, "b_i0": torch.zeros(64, device="cuda"), "W_i1": draw(d, 64) * 0.1, "b_i1": torch.zeros(d, device="cuda"),
         "bridges": draw(nb, d)}
    ctx.load_item_weights(w)
    for n in (1, 15, 16, 17, 257, M):
        raw, iid = draw(n, 64), draw(n, d)
        ctx.item_nearline_compute(None, raw, iid)
        if nb % 2 == 0:
            out = torch.empty(n, nb, dtype=torch.bfloat16, device="cuda")
            ctx.gather_sidecars(torch.arange(n, dtype=torch.int32, device="cuda"), out)
            got = out.float().cpu()
        else:
            got = _bridge_weights_by_scoring(ctx, n)
        want = orc.item_nearline(orc.BF16, I_id=iid.cpu().view(torch.int16).numpy().view(np.uint16),
                                 bridges=w["bridges"].cpu().view(torch.int16).numpy().view(np.uint16))["w_hat"]
        assert np.abs(got.numpy() - want).max() <= 2.0 ** -9
        assert ctx.poll_status() == 0
    ctx.close()


@pytest.mark.parametrize("d,dU", [(128, 128), (64, 256), (256, 64), (256, 256), (128, 96)])
def test_user_side_at_the_lengths_around_its_row_and_key_steps(d, dU):
    """Eqs. 1-3 from raw features: sequence lengths around the 16 rows of a product, the keys of a profile step (32, 16 or 8)
    and the 128-key blocks; widths of every product and one that takes the CUDA cores.  u and p_u carry bf16 S and attention
    rows (2^-9 relative on values below 0.1), S one rounding."""
    wl = helpers.MINI["c2"].with_(name=f"user_edges_{d}_{dU}", d=d, dU=dU, M=500, N=50, L=300, mini_batch=0)
    weights = synth.make_weights(wl, zero_bias=False)
    srv = serving.Server(wl, weights, synth.make_item_table(wl))
    oracle = helpers.make_oracle(wl, weights, M=500)
    W1 = synth.as_f32(weights["mlp"]["W"][0], wl.dtype).astype(np.float64)
    for L in (1, 7, 16, 17, 33, 128, 300):
        rq = synth.make_request(wl, L, L=L)
        st = srv.precompute(L, srv.upload_request(rq, B.USER_RAW))
        u, S, pu = srv.ctx.user_state_export(st, L)
        torch.cuda.synchronize()
        u_ref, S_ref = oracle.user_state(rq["profile"], rq["seq"])
        assert np.abs(S.float().cpu().numpy() - S_ref).max() <= TOL
        assert np.abs(u.cpu().numpy() - u_ref).max() <= TOL
        assert np.abs(pu.cpu().numpy() - (W1[:, :d] @ u_ref + weights["mlp"]["b"][0])).max() <= TOL
        st.release()
    assert srv.ctx.poll_status() == 0
    srv.close()


@pytest.mark.parametrize("n_bridge", [3, 16])
@pytest.mark.parametrize("base", ["c2", "c5"])
def test_bridge_embedding_columns_around_half_a_tile(base, n_bridge):
    """v = w^ V for candidate counts around the 64 of a block, one and several requests, with and without mini-batches."""
    wl = helpers.MINI[base].with_(name=f"bea_edges_{base}_{n_bridge}", R=3, N=200, M=2000, L=40, mini_batch=70 if base == "c2" else 0,
                                  blocks=synth.BLK_CROSS | synth.BLK_BEA, n_bridge=n_bridge)
    weights, table = synth.make_weights(wl, zero_bias=False), synth.make_item_table(wl)
    srv, oracle = serving.Server(wl, weights, table), helpers.make_oracle(wl, weights, M=wl.M)
    rqs = [synth.make_request(wl, r) for r in range(3)]
    states = [srv.precompute(r, srv.upload_request(rq, B.USER_PROJECTED)) for r, rq in enumerate(rqs)]
    g = np.random.default_rng(9)
    for sizes in ((1, 64, 65), (63, 128, 200)):
        lists = [g.choice(wl.M, n, replace=False).astype(np.int32) for n in sizes]
        lists[2][5] = wl.M
        want = [oracle.score(table, helpers.projected_request(wl, rq), ids) for rq, ids in zip(rqs, lists)]
        for got, w in zip(srv.score_many(states, lists), want):
            _check(got, w)
        _check(srv.score_ids(states[2], lists[2]), want[2])
    assert srv.ctx.poll_status() == B.STATUS_BAD_ID
    srv.close()


@pytest.mark.parametrize("F,dc,hidden", [(16, 8, (256, 128)), (8, 16, (512, 80)), (2, 32, (64,)), (3, 64, (1024, 64, 16)), (1, 128, (256, 192)),
                                         (4, 32, (768, 256, 48))])
def test_layer_kernel_over_the_field_widths_and_slices_it_accepts(F, dc, hidden):
    """The layer kernel on CTA pairs: one, two, four and eight fields per 64-column chunk and fields over several chunks; one to
    four output slices, slices rounded up to 64 columns; one tile alone, an odd number of tiles, ragged tiles; ids outside the
    table."""
    wl = helpers.MINI["c3"].with_(name=f"layers_{F}_{dc}_{len(hidden)}", R=3, N=400, M=3000, L=260, F=F, dc=dc, B=300, hidden=hidden,
                                  bucket_mode=synth.BUCKET_HASH)
    weights, table = synth.make_weights(wl, zero_bias=False), synth.make_item_table(wl)
    srv, oracle = serving.Server(wl, weights, table), helpers.make_oracle(wl, weights, M=wl.M)
    rqs = [synth.make_request(wl, r) for r in range(3)]
    states = [srv.precompute(r, srv.upload_request(rq, B.USER_PROJECTED)) for r, rq in enumerate(rqs)]
    g = np.random.default_rng(4)
    for sizes in ((1, 128, 129), (256, 31, 400)):
        lists = [g.choice(wl.M, n, replace=False).astype(np.int32) for n in sizes]
        lists[2][7] = -3
        want = [oracle.score(table, helpers.projected_request(wl, rq), ids) for rq, ids in zip(rqs, lists)]
        for got, w in zip(srv.score_many(states, lists), want):
            _check(got, w)
        for st, ids, w in zip(states, lists, want):
            _check(srv.score_ids(st, ids), w)
    assert srv.ctx.poll_status() == B.STATUS_BAD_ID
    srv.close()


def test_layer_kernel_with_several_items_per_pair():
    """More pairs of tiles than the GPU has pairs of SMs, four slices each: accumulators and ring stages in every phase, checked
    on the candidates around the tile edges of a few requests."""
    wl = helpers.MINI["c5"].with_(name="layers_many", R=12, N=1700, M=4000, L=20, F=4, B=64)
    weights, table = synth.make_weights(wl, zero_bias=False), synth.make_item_table(wl)
    srv, oracle = serving.Server(wl, weights, table), helpers.make_oracle(wl, weights, M=wl.M)
    rqs = [synth.make_request(wl, r) for r in range(wl.R)]
    states = [srv.precompute(r, srv.upload_request(rq, B.USER_PROJECTED)) for r, rq in enumerate(rqs)]
    g = np.random.default_rng(6)
    lists = [g.choice(wl.M, 1700 - 13 * r, replace=False).astype(np.int32) for r in range(wl.R)]
    got = srv.score_many(states, lists)
    for r in (0, 5, 11):
        n = len(lists[r])
        at = np.unique(np.clip(np.concatenate([np.arange(0, n, 128), np.arange(127, n, 128), [n - 1], g.integers(0, n, 40)]), 0, n - 1))
        _check(got[r][at], oracle.score(table, helpers.projected_request(wl, rqs[r]), lists[r][at]))
    assert srv.ctx.poll_status() == 0
    srv.close()


@pytest.mark.parametrize("base", ["c2", "c5"])
@pytest.mark.parametrize("blocks", [synth.BLK_ATT | synth.BLK_CROSS, synth.BLK_CROSS | synth.BLK_LSH_DIN | synth.BLK_SIMTIER, helpers.ALL_BLOCKS])
def test_key_ranges_split_over_ctas(base, blocks):
    """Few tiles with many keys: every tile's keys in pieces on CTAs of their own, joined by a launch that follows.  Requests of 1
    to 3000 items in one launch (tiles with fewer key blocks than pieces among them), ragged tiles, bad ids, twice in a row,
    and each request by itself."""
    wl = helpers.MINI[base].with_(name=f"split_{base}_{blocks}", R=4, N=130, M=2000, L=3000, F=2, B=64, mini_batch=0, blocks=blocks, n_tiers=9)
    weights, table = synth.make_weights(wl, zero_bias=False), synth.make_item_table(wl)
    srv, oracle = serving.Server(wl, weights, table), helpers.make_oracle(wl, weights, M=wl.M)
    rqs = [synth.make_request(wl, r, L=L) for r, L in enumerate((3000, 1, 129, 1500))]
    states = [srv.precompute(r, srv.upload_request(rq, B.USER_PROJECTED)) for r, rq in enumerate(rqs)]
    g = np.random.default_rng(8)
    lists = [g.choice(wl.M, n, replace=False).astype(np.int32) for n in (130, 5, 128, 1)]
    lists[0][11] = wl.M
    want = [oracle.score(table, helpers.projected_request(wl, rq), ids) for rq, ids in zip(rqs, lists)]
    first = srv.score_many(states, lists)
    again = srv.score_many(states, lists)
    for got, rep, w, st, ids in zip(first, again, want, states, lists):
        _check(got, w)
        assert np.array_equal(got, rep, equal_nan=True)
        _check(srv.score_ids(st, ids), w)
    assert srv.ctx.poll_status() == B.STATUS_BAD_ID
    srv.close()


@pytest.mark.parametrize("s_scale", [1.0, 1024.0])
def test_split_pieces_with_and_without_a_running_maximum(s_scale):
    """Sequence rows so large that every piece keeps a maximum of its own: the pieces are joined at different exponent offsets.
    Inputs 1024 times off the workload's distribution leave attention rows of that magnitude, rounded to bf16 (2^-9 relative):
    1e-2 of the largest logit, as for the unsplit kernel."""
    wl = helpers.MINI["c2"].with_(name="split_sharp", R=1, N=200, M=2000, L=2500, F=2, B=64, mini_batch=0)
    weights, table = synth.make_weights(wl, zero_bias=False), synth.make_item_table(wl)
    rq = synth.make_request(wl, 0)
    rq["S"] = synth.store(synth.as_f32(rq["S"], wl.dtype) * np.float32(s_scale), wl.dtype)
    srv, oracle = serving.Server(wl, weights, table), helpers.make_oracle(wl, weights, M=wl.M)
    st = srv.precompute(0, srv.upload_request(rq, B.USER_PROJECTED))
    ids = np.random.default_rng(3).choice(wl.M, 200, replace=False).astype(np.int32)
    want = oracle.score(table, helpers.projected_request(wl, rq), ids)
    _check(srv.score_ids(st, ids), want, TOL if s_scale == 1.0 else 1e-2 * max(1.0, np.abs(want).max()))
    assert srv.ctx.poll_status() == 0
    srv.close()


@pytest.mark.parametrize("n_cat", [3, 1500])
def test_category_jobs_over_one_and_several_batches_of_groups(n_cat):
    """Sub-sequences cut into pieces, among them long, short and empty ones: few categories (every tile split) and more groups than
    the placing block has threads (two requests x 1500 categories)."""
    wl = helpers.MINI["c2"].with_(name=f"sim_jobs_{n_cat}", R=2, N=600, M=4000, L=6000, F=2, B=64, mini_batch=0, n_categories=n_cat,
                                  blocks=synth.BLK_ATT | synth.BLK_CROSS | synth.BLK_LSH_DIN | synth.BLK_SIMTIER)
    weights, table = synth.make_weights(wl, zero_bias=False), synth.make_item_table(wl)
    srv, oracle = serving.Server(wl, weights, table), helpers.make_oracle(wl, weights, M=wl.M)
    rqs = [synth.make_request(wl, r) for r in range(2)]
    states = [srv.precompute(r, srv.upload_request(rq, B.USER_PROJECTED)) for r, rq in enumerate(rqs)]
    g = np.random.default_rng(2)
    lists = [g.choice(wl.M, n, replace=False).astype(np.int32) for n in (600, 333)]
    want = [oracle.score(table, helpers.projected_request(wl, rq), ids) for rq, ids in zip(rqs, lists)]
    for got, w in zip(srv.score_many(states, lists), want):
        _check(got, w)
    _check(srv.score_ids(states[1], lists[1]), want[1])
    assert srv.ctx.poll_status() == 0
    srv.close()


@pytest.mark.parametrize("dtype,d,hidden,F,dc,blocks", [
    ("f32", 64, (256, 128), 8, 16, helpers.ALL_BLOCKS), ("f32", 32, (264, 8), 3, 8, synth.BLK_ATT | synth.BLK_CROSS),
    ("f32", 96, (1024, 40, 520), 5, 24, helpers.ALL_BLOCKS), ("f32", 256, (8,), 2, 8, synth.BLK_CROSS | synth.BLK_LSH_DIN | synth.BLK_SIMTIER),
    ("bf16", 160, (72, 264), 4, 8, helpers.ALL_BLOCKS), ("bf16", 224, (1000,), 1, 8, synth.BLK_ATT),
    ("f32", 32, (64, 32), 256, 16, synth.BLK_ATT | synth.BLK_CROSS), ("f32", 32, (32, 16), 256, 24, synth.BLK_ATT | synth.BLK_CROSS | synth.BLK_LSH_DIN)])
def test_cuda_core_scoring_over_widths_and_sequence_lengths(dtype, d, hidden, F, dc, blocks):
    """The CUDA-core kernel: sequence lengths around its 32-key chunks, layers narrower than a warp's outputs, of whole and of partial
    column blocks, inputs too wide for the weight ring and for the key chunks (the last two rows); every d it accepts a step of."""
    wl = synth.C1.with_(name=f"simt_{dtype}_{d}_{len(hidden)}_{F}", dtype=dtype, d=d, hidden=hidden, F=F, dc=dc, B=16, R=1, N=75, M=800, L=160, blocks=blocks,
                        emit_sigmoid=0, lsh_din_norm=synth.NORM_MEAN, simtier_norm=synth.NORM_MEAN, mini_batch=30, bucket_mode=synth.BUCKET_HASH)
    weights, table = synth.make_weights(wl, zero_bias=False), synth.make_item_table(wl)
    srv, oracle = serving.Server(wl, weights, table, path=B.PATH_SIMT), helpers.make_oracle(wl, weights, M=wl.M)
    ids = np.random.default_rng(1).choice(wl.M, 75, replace=False).astype(np.int32)
    ids[9] = -1
    for L in (1, 31, 32, 33, 64, 65, 101, 160):
        rq = synth.make_request(wl, L, L=L)
        st = srv.precompute(L, srv.upload_request(rq, B.USER_PROJECTED))
        want = oracle.score(table, helpers.projected_request(wl, rq), ids)
        # fp32 arithmetic throughout (sums of up to 6500 terms: 1e-5 of the largest logit where that exceeds 1); bf16 storage as elsewhere
        _check(srv.score_ids(st, ids), want, 1e-5 * max(1.0, np.nanmax(np.abs(want))) if dtype == "f32" else TOL)
        st.release()
    assert srv.ctx.poll_status() == B.STATUS_BAD_ID
    srv.close()


@pytest.mark.parametrize("mini_batch", [0, 50, 128])
def test_category_rows_in_whole_tiles_of_their_requests(mini_batch):
    """Categories of a few candidates each, every block on: the kernels that do not depend on the category take the grouped
    candidates of a request in whole tiles, whatever the mini-batch; requests of one and of several tiles, ids outside the table."""
    wl = helpers.MINI["c2"].with_(name=f"sim_rows_{mini_batch}", R=3, N=600, M=4000, L=900, F=2, B=64, mini_batch=mini_batch, n_categories=40,
                                  blocks=helpers.ALL_BLOCKS)
    weights, table = synth.make_weights(wl, zero_bias=False), synth.make_item_table(wl)
    srv, oracle = serving.Server(wl, weights, table), helpers.make_oracle(wl, weights, M=wl.M)
    rqs = [synth.make_request(wl, r) for r in range(3)]
    states = [srv.precompute(r, srv.upload_request(rq, B.USER_PROJECTED)) for r, rq in enumerate(rqs)]
    g = np.random.default_rng(4)
    lists = [g.choice(wl.M, n, replace=False).astype(np.int32) for n in (600, 1, 333)]
    lists[2][7], lists[2][300] = -1, wl.M
    want = [oracle.score(table, helpers.projected_request(wl, rq), ids) for rq, ids in zip(rqs, lists)]
    for got, w in zip(srv.score_many(states, lists), want):
        _check(got, w)
    for i in (0, 2):
        _check(srv.score_ids(states[i], lists[i]), want[i])
    assert srv.ctx.poll_status() == B.STATUS_BAD_ID
    srv.close()


@pytest.mark.parametrize("dI,hI,d", [(64, 64, 64), (128, 192, 128), (512, 256, 128)])
def test_item_tower_over_its_pairs_of_tiles_and_both_buffers(dI, hI, d):
    """The one-kernel tower: rows that fill no tile, one tile of a pair, a pair, one item per pair of SMs and one or two more (both
    buffers, first use and re-use), one and eight K chunks.  bf16 has eight significant bits, so rounding a hidden activation, and the
    row, moves it by up to 2^-8 of itself (half of the last bit, 2^-7, just above a power of two): 2^-8 of the sum of the absolute
    terms, and of the row and that sum's share of it; 1e-4 covers the fp32 sums of up to 512 terms of order 1."""
    M = 74 * 256 * 2 + 129
    ctx = B.Aif(B.make_config(dtype=B.BF16, M=M, d=d, L_max=8, hidden=(64,), blocks=B.BLK_BEA, n_bridge=2))
    g = torch.Generator(device="cuda").manual_seed(dI)

    def draw(*shape):
        return torch.randn(*shape, generator=g, device="cuda").to(torch.bfloat16)

    w = {"W_i0": draw(hI, dI) * 0.1, "b_i0": torch.randn(hI, generator=g, device="cuda"), "W_i1": draw(d, hI) * 0.1,
         "b_i1": torch.randn(d, generator=g, device="cuda"), "bridges": draw(2, d)}
    ctx.load_item_weights(w)
    raw = draw(M, dI)
    for n in (1, 128, 129, 256, 257, 74 * 256, 74 * 256 + 1, M):
        ctx.item_nearline_compute(None, raw[:n], draw(n, d))
        out = torch.empty(n, d, dtype=torch.bfloat16, device="cuda")
        ctx.gather_rows(torch.arange(n, dtype=torch.int32, device="cuda"), out)
        h = torch.relu(raw[:n].double() @ w["W_i0"].double().T + w["b_i0"].double())
        want = h @ w["W_i1"].double().T + w["b_i1"].double()
        moved = 2.0 ** -8 * (h @ w["W_i1"].double().abs().T)
        bound = moved + 2.0 ** -8 * (want.abs() + moved) + 1e-4
        ratio = (out.double() - want).abs() / bound
        assert ratio.max().item() <= 1.0, f"n {n}: {int((ratio > 1).sum())} elements, worst {ratio.max().item():.2f} of the bound at {divmod(int(ratio.argmax()), d)}"
        assert ctx.poll_status() == 0
    ctx.close()


@pytest.mark.parametrize("H2,F,dc", [(64, 4, 16), (192, 2, 64), (256, 16, 32)])
def test_whole_mlp_in_one_kernel_at_the_edges_of_its_range(H2, F, dc):
    """Two layers of 512 and at most 256 units, all tiles at once: one tile (the pair's other tile does not exist), odd and even numbers
    of tiles, the last number it takes and the first it does not (148 and 149), two requests whose tiles share a pair."""
    wl = helpers.MINI["c2"].with_(name=f"mlp_{H2}_{F}_{dc}", R=2, N=148 * 128 + 1, M=20000, L=300, mini_batch=0, hidden=(512, H2), F=F, dc=dc, B=64,
                                  blocks=helpers.ALL_BLOCKS)
    weights, table = synth.make_weights(wl, zero_bias=False), synth.make_item_table(wl)
    srv, oracle = serving.Server(wl, weights, table), helpers.make_oracle(wl, weights, M=wl.M)
    rqs = [synth.make_request(wl, r) for r in range(2)]
    states = [srv.precompute(r, srv.upload_request(rq, B.USER_PROJECTED)) for r, rq in enumerate(rqs)]
    g = np.random.default_rng(6)
    ids = g.choice(wl.M, wl.N, replace=False).astype(np.int32)
    ids[3] = -1
    pick = np.unique(np.concatenate([g.choice(wl.N, 60), [0, 3, 127, 128, 255, 256, wl.N - 2, wl.N - 1]]))
    want = oracle.score(table, helpers.projected_request(wl, rqs[0]), ids[pick])
    for n in (1, 128, 129, 300, 147 * 128, 148 * 128, 148 * 128 + 1):
        got = srv.score_ids(states[0], ids[:n])
        _check(got[pick[pick < n]], want[pick < n])
    a, b = ids[:200], ids[500:611]
    for got, rq, i in zip(srv.score_many(states, [a, b]), rqs, (a, b)):
        _check(got, oracle.score(table, helpers.projected_request(wl, rq), i))
    assert srv.ctx.poll_status() == B.STATUS_BAD_ID
    srv.close()


@pytest.mark.parametrize("dtype,d,hidden", [("bf16", 256, (1024, 512, 256)), ("bf16", 128, (512, 256)), ("bf16", 64, (72,)), ("f32", 256, (264, 8)), ("f32", 32, (8,))])
def test_the_users_share_of_the_first_layer_is_one_running_sum(dtype, d, hidden):
    """p_u[j] = b1[j], then one multiply-add per column of u in their order: bit for bit, whatever the number of columns and units
    (products of bf16 values are exact in fp32; fp32 ones, and their sums, are formed in 80 bits and rounded to fp32 once)."""
    wl = synth.C2.with_(name=f"pu_{dtype}_{d}_{len(hidden)}", dtype=dtype, d=d, hidden=hidden, F=2, dc=32, B=16, R=1, N=10, M=500, L=20, mini_batch=0)
    weights = synth.make_weights(wl, zero_bias=False)
    srv = serving.Server(wl, weights, synth.make_item_table(wl))
    rq = synth.make_request(wl, 0)
    st = srv.precompute(0, srv.upload_request(rq, B.USER_PROJECTED))
    u, _, pu = srv.ctx.user_state_export(st, wl.L)
    u_in, W1 = synth.as_f32(rq["u"], dtype), synth.as_f32(weights["mlp"]["W"][0], dtype)
    want = weights["mlp"]["b"][0].astype(np.float32)
    for k in range(d):
        want = (want.astype(np.longdouble) + u_in[k].astype(np.longdouble) * W1[:, k].astype(np.longdouble)).astype(np.float32)
    assert np.array_equal(u.cpu().numpy(), u_in)
    assert np.array_equal(pu.cpu().numpy(), want)
    assert srv.ctx.poll_status() == 0
    srv.close()


def _overflow_request(wl, minus_inf):
    """A projected request whose scores are minus infinity for the given keys against an item whose first column is 2^80 (the
    product overflows fp32), and that column's share is zero for all others."""
    rq = synth.make_request(wl, 0)
    S = synth.as_f32(rq["S"], wl.dtype).copy()
    S[:, 0] = 0.0
    S[minus_inf, 0] = -(2.0 ** 80)
    rq["S"] = synth.store(S, wl.dtype)
    return rq


@pytest.mark.parametrize("base,n_cat", [("c2", 0), ("c5", 0), ("c2", 1)])
def test_split_pieces_that_hold_nothing_but_minus_infinity(base, n_cat):
    """Keys whose scores overflow to minus infinity carry no weight, also where they are all that a piece of the keys holds: the
    pieces' join gives what the other pieces say.  The layers do not read the column that overflows."""
    wl = helpers.MINI[base].with_(name=f"split_inf_{base}_{n_cat}", R=1, N=100, M=300, L=2560, F=2, B=64, mini_batch=0, n_categories=n_cat,
                                  blocks=synth.BLK_ATT | synth.BLK_CROSS)
    weights, table = synth.make_weights(wl, zero_bias=False), synth.make_item_table(wl)
    E = synth.as_f32(table["E"], wl.dtype).copy()
    E[:, 0] = 2.0 ** 80
    table["E"] = synth.store(E, wl.dtype)
    weights["mlp"]["W"][0][:, wl.d] = 0
    rq = _overflow_request(wl, slice(1280, 2560))
    if n_cat:
        rq["seq_cat"] = np.zeros(wl.L, dtype=np.int32)
    srv, oracle = serving.Server(wl, weights, table), helpers.make_oracle(wl, weights, M=wl.M)
    st = srv.precompute(0, srv.upload_request(rq, B.USER_PROJECTED))
    ids = np.random.default_rng(3).choice(wl.M, 100, replace=False).astype(np.int32)
    want = oracle.score(table, helpers.projected_request(wl, rq), ids)
    assert np.isfinite(want).all()
    _check(srv.score_ids(st, ids), want)
    assert srv.ctx.poll_status() == 0
    srv.close()


@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("bf16", 256), ("bf16", 64), ("f32", 64), ("f32", 128)])
def test_profile_attention_where_a_slice_holds_nothing_but_minus_infinity(dtype, d):
    """Eq. 3 with scores that overflow to minus infinity for a whole step of keys (32, 16 or 8 by width), between keys that have the
    weight: those keys have none.  Identity projections, so that S and the projected profile are the inputs."""
    step = 8 * (4 if d <= 64 else 2 if d <= 128 else 1)
    wl = synth.C2.with_(name=f"prof_inf_{dtype}_{d}", dtype=dtype, d=d, dU=d, hidden=(64,), F=2, dc=32, B=16, R=1, N=10, M=500, L=96, mini_batch=0)
    weights = synth.make_weights(wl, zero_bias=False)
    eye = synth.store(np.eye(d, dtype=np.float32), dtype)
    weights["user"]["W_seq"], weights["user"]["W_profile"] = eye, eye.copy()
    rq = synth.make_request(wl, 0)
    seq, prof = synth.as_f32(rq["seq"], dtype).copy(), synth.as_f32(rq["profile"], dtype).copy()
    prof[0] = 2.0 ** 122
    seq[:, 0] = 0.0
    seq[32:32 + step, 0] = -1024.0
    rq["seq"], rq["profile"] = synth.store(seq, dtype), synth.store(prof, dtype)
    srv, oracle = serving.Server(wl, weights, synth.make_item_table(wl)), helpers.make_oracle(wl, weights, M=wl.M)
    st = srv.precompute(0, srv.upload_request(rq, B.USER_RAW))
    u, _, _ = srv.ctx.user_state_export(st, wl.L)
    u_ref, _ = oracle.user_state(rq["profile"], rq["seq"])
    assert np.isfinite(u_ref).all()
    # attention rows of size 10^3, rounded to bf16 where the storage is (2^-9), through a layer of order-1 weights
    assert np.abs(u.cpu().numpy() - u_ref).max() <= (1e-2 if dtype == "bf16" else 1e-5) * np.abs(u_ref).max()
    assert srv.ctx.poll_status() == 0
    srv.close()


def _host_workload(kind):
    if kind == "fused":
        return helpers.MINI["c2"].with_(name="host_fused", R=2, N=300, M=4000, L=100, mini_batch=0)
    if kind == "chain":
        return helpers.MINI["c3"].with_(name="host_chain", R=2, N=300, M=4000, L=300)
    if kind == "no_cross":
        return helpers.MINI["c2"].with_(name="host_no_cross", R=2, N=300, M=4000, L=300, mini_batch=0, blocks=synth.BLK_ATT)
    if kind == "categories":
        return helpers.MINI["c2"].with_(name="host_cat", R=2, N=300, M=4000, L=900, F=2, B=64, mini_batch=0, n_categories=7, blocks=helpers.ALL_BLOCKS)
    return helpers.MINI["c1"].with_(name="host_simt", R=2, N=300, M=4000)


@pytest.mark.parametrize("kind", ["fused", "chain", "no_cross", "categories", "simt"])
def test_host_buffers_page_locked_pageable_and_one_of_each(kind):
    """Ids read across the bus by a scoring kernel, by a copy kernel, or copied; logits stored across the bus or copied back; logits
    written over the ids they belong to: the device buffers' result, bit for bit, on every scoring path, for one request and several."""
    wl = _host_workload(kind)
    weights, table = synth.make_weights(wl, zero_bias=False), synth.make_item_table(wl)
    srv = serving.Server(wl, weights, table)
    states = [srv.precompute(r, srv.upload_request(synth.make_request(wl, r), B.USER_PROJECTED)) for r in range(2)]
    g = np.random.default_rng(5)
    lists = [g.choice(wl.M, n, replace=False).astype(np.int32) for n in (300, 37)]
    lists[0][8] = -1
    want, one = np.concatenate(srv.score_many(states, lists)), srv.score_ids(states[0], lists[0])
    all_ids, offs = np.concatenate(lists), [0, 300, 337]
    for ids_pinned in (True, False):
        for out_pinned in (True, False):
            ids, out = torch.from_numpy(all_ids.copy()), torch.full((337,), -7.0)
            ids, out = ids.pin_memory() if ids_pinned else ids, out.pin_memory() if out_pinned else out
            srv.ctx.score_batch_host(states, ids, offs, out)
            assert np.array_equal(out.numpy(), want, equal_nan=True)
            out.fill_(-7.0)
            srv.ctx.score_host(states[0], ids[:300], out[:300])
            assert np.array_equal(out[:300].numpy(), one, equal_nan=True) and (out[300:] == -7.0).all()
    for pinned in (True, False):
        for batch in (True, False):
            buf = torch.from_numpy(all_ids.copy())
            buf = buf.pin_memory() if pinned else buf
            if batch:
                srv.ctx.score_batch_host(states, buf, offs, buf.view(torch.float32))
                assert np.array_equal(buf.view(torch.float32).numpy(), want, equal_nan=True)
            else:
                srv.ctx.score_host(states[0], buf[:300], buf.view(torch.float32)[:300])
                assert np.array_equal(buf.view(torch.float32)[:300].numpy(), one, equal_nan=True) and np.array_equal(buf[300:].numpy(), lists[1])
    assert srv.ctx.poll_status() == B.STATUS_BAD_ID
    srv.close()


@pytest.mark.parametrize("n", [8192, 8193])
def test_host_batches_around_the_number_of_ids_read_across_the_bus(n):
    """Up to 65536 page-locked ids are read by the kernels, longer lists are copied; the logits go straight to host memory either way."""
    wl = helpers.MINI["c2"].with_(name=f"host_big_{n}", R=8, N=n, M=20000, L=20, mini_batch=0)
    srv = serving.Server(wl, synth.make_weights(wl), synth.make_item_table(wl))
    states = [srv.precompute(r, srv.upload_request(synth.make_request(wl, r), B.USER_PROJECTED)) for r in range(8)]
    g = np.random.default_rng(5)
    lists = [g.choice(wl.M, n, replace=False).astype(np.int32) for _ in range(8)]
    want = np.concatenate(srv.score_many(states, lists))
    ids, out = torch.from_numpy(np.concatenate(lists)).pin_memory(), torch.full((8 * n,), -7.0).pin_memory()
    srv.ctx.score_batch_host(states, ids, [n * r for r in range(9)], out)
    assert np.array_equal(out.numpy(), want)
    assert srv.ctx.poll_status() == 0
    srv.close()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_cuda_core_scoring_at_the_widest_input_that_fits_shared_memory(dtype):
    """One cross field so wide that input, activations and item vectors all but fill shared memory: accepted, and right; eight columns
    more are refused without harm."""
    # 8 candidates of (k1 + d + 2 H) floats and 24 words per candidate: 227 KB holds 7240 columns, units and tier counts in all
    wl = synth.C1.with_(name=f"widest_{dtype}", dtype=dtype, d=32, hidden=(8,), F=1, dc=7152, B=4, R=1, N=20, M=100, L=5, mini_batch=0, emit_sigmoid=0,
                        blocks=synth.BLK_CROSS | synth.BLK_SIMTIER, n_tiers=5, simtier_norm=synth.NORM_MEAN, bucket_mode=synth.BUCKET_HASH)
    for more, fits in ((0, True), (8, False)):
        w = wl.with_(dc=wl.dc + more)
        weights, table = synth.make_weights(w, zero_bias=False), synth.make_item_table(w)
        srv, oracle = serving.Server(w, weights, table, path=B.PATH_SIMT), helpers.make_oracle(w, weights, M=w.M)
        rq = synth.make_request(w, 0)
        st = srv.precompute(0, srv.upload_request(rq, B.USER_PROJECTED))
        ids = np.arange(20, dtype=np.int32)
        if fits:
            want = oracle.score(table, helpers.projected_request(w, rq), ids)
            _check(srv.score_ids(st, ids), want, 1e-5 * max(1.0, np.abs(want).max()) if dtype == "f32" else TOL)
        else:
            with pytest.raises(B.AifError):
                srv.score_ids(st, ids)
        assert srv.ctx.poll_status() == 0
        srv.close()


@pytest.mark.parametrize("dtype,d,hidden,F,dc", [("f32", 32, (16,), 2, 8), ("f32", 64, (256, 128), 40, 8), ("bf16", 96, (264, 64), 33, 16), ("f32", 256, (520, 256), 3, 24), ("f32", 64, (192, 40), 9, 8)])
def test_cuda_core_scoring_of_more_candidates_than_one_block_per_sm(dtype, d, hidden, F, dc):
    """Launches of up to two blocks per SM and of more take different forms of the kernel: the candidates around the change, fields in
    more than one group of 32, one and several requests; both forms agree with the oracle and, bit for bit, with each other."""
    wl = synth.C1.with_(name=f"simt_many_{dtype}_{d}_{F}", dtype=dtype, d=d, hidden=hidden, F=F, dc=dc, B=16, R=2, N=296 * 8 + 9, M=3000, L=70, emit_sigmoid=0,
                        blocks=helpers.ALL_BLOCKS, lsh_din_norm=synth.NORM_MEAN, simtier_norm=synth.NORM_MEAN, mini_batch=0, bucket_mode=synth.BUCKET_HASH)
    weights, table = synth.make_weights(wl, zero_bias=False), synth.make_item_table(wl)
    srv, oracle = serving.Server(wl, weights, table, path=B.PATH_SIMT), helpers.make_oracle(wl, weights, M=wl.M)
    rqs = [synth.make_request(wl, r, L=L) for r, L in enumerate((70, 33))]
    states = [srv.precompute(r, srv.upload_request(rq, B.USER_PROJECTED)) for r, rq in enumerate(rqs)]
    ids = np.random.default_rng(1).choice(wl.M, wl.N, replace=False).astype(np.int32)
    ids[9] = -1
    pick = np.unique(np.concatenate([[0, 7, 8, 9, wl.N - 1, wl.N - 10], np.random.default_rng(2).choice(wl.N, 60)]))
    wants = [oracle.score(table, helpers.projected_request(wl, rq), ids[pick]) for rq in rqs]
    # sums of up to 1500 terms in fp32; bf16 storage as elsewhere
    tol = 1e-5 * max(1.0, np.nanmax(np.abs(wants[0]))) if dtype == "f32" else TOL
    for n in (296 * 8, 296 * 8 + 1, wl.N):
        got = srv.score_ids(states[0], ids[:n])
        _check(got[pick[pick < n]], wants[0][pick < n], tol)
    parts = np.concatenate([srv.score_ids(states[0], ids[:1200]), srv.score_ids(states[0], ids[1200:])])
    assert np.array_equal(got, parts, equal_nan=True)    # a candidate's logit does not depend on how many others there are
    for got, w in zip(srv.score_many(states, [ids, ids]), wants):
        _check(got[pick], w, tol)
    assert srv.ctx.poll_status() == B.STATUS_BAD_ID
    srv.close()


@pytest.mark.parametrize("Bk", [1, 3, 255, 1000, 4096, 32769, 65534])
def test_buckets_of_the_kernel_chain_for_numbers_that_are_no_power_of_two(Bk):
    """The hash modulo the number of buckets, by a multiplication where that is no power of two: the smallest and the largest number,
    and numbers around powers of two; a wrong bucket is another embedding, 0.1 in a logit."""
    wl = helpers.MINI["c3"].with_(name=f"buckets_{Bk}", R=1, N=4000, M=30000, L=5, F=2, dc=32, B=Bk, hidden=(256, 64), blocks=synth.BLK_CROSS,
                                  bucket_mode=synth.BUCKET_HASH, sigma=0.5)
    weights, table = synth.make_weights(wl, zero_bias=False), synth.make_item_table(wl)
    srv, oracle = serving.Server(wl, weights, table), helpers.make_oracle(wl, weights, M=wl.M)
    rq = synth.make_request(wl, 0)
    st = srv.precompute(0, srv.upload_request(rq, B.USER_PROJECTED))
    ids = np.random.default_rng(3).choice(wl.M, wl.N, replace=False).astype(np.int32)
    want = oracle.score(table, helpers.projected_request(wl, rq), ids)
    # activations of order 1: bf16 budget of the largest logit
    _check(srv.score_ids(st, ids), want, 1e-2 * max(1.0, np.abs(want).max()))
    assert srv.ctx.poll_status() == 0
    srv.close()


@pytest.mark.parametrize("d,L_max,n_cat,most", [(128, 1, 0, 16), (128, 128, 0, 16), (256, 64, 0, 24), (128, 512, 3, 40), (128, 300, 0, 60)])
def test_contexts_take_no_more_room_for_partial_results_than_their_sequences_can_use(d, L_max, n_cat, most):
    """A context whose sequences are one key block (one that only holds a table among them) never splits keys, and few tiles have few
    pieces: megabytes in all for a table of 1000 items and 128 candidates, every block on."""
    cfg = B.make_config(dtype=B.BF16, M=1000, d=d, L_max=L_max, hidden=(64,), F=2, B=16, dc=32, n_categories=n_cat, blocks=helpers.ALL_BLOCKS,
                        max_batch_candidates=128, max_user_states=1)
    ctx = B.Aif(cfg)
    assert ctx.get_stats().device_bytes <= most << 20
    ctx.close()


@pytest.mark.parametrize("H2,L", [(256, 200), (64, 128), (192, 129), (256, 1)])
def test_small_requests_at_the_edges_of_their_tiles(H2, L):
    """Requests by themselves go in tiles of 16, 32 or 48 candidates on clusters of four CTAs, larger ones by the kernel of one CTA per tile:
    numbers of candidates on either side of every change, an id outside the table among them, and the widths of the second layer that
    a cluster splits into quarters of 16 to 64 units."""
    sizes = [1, 15, 16, 17, 33, 560, 577, 592, 593, 1000, 1153, 1185, 1729, 1777, 1900]
    wl = helpers.MINI["c2"].with_(name=f"split_{H2}_{L}", N=max(sizes), M=20_000, mini_batch=0, L=L, hidden=(512, H2))
    weights, table = synth.make_weights(wl, zero_bias=False), synth.make_item_table(wl)
    srv = serving.Server(wl, weights, table, path=B.PATH_TENSOR)
    oracle = helpers.make_oracle(wl, weights, M=wl.M)
    rq = synth.make_request(wl, 0)
    st = srv.precompute(0, srv.upload_request(rq, B.USER_PROJECTED))
    sampler = synth.IdSampler(wl)
    for n in sizes:
        ids = sampler.request_ids(0, n)
        if n > 20:
            ids[n // 2] = wl.M
        got = srv.score_ids(st, ids)
        pick = np.unique(np.r_[0:min(n, 50), max(0, n - 50):n, n // 2])
        _check(got[pick], oracle.score(table, helpers.projected_request(wl, rq), ids[pick]))
        assert int(np.isnan(got).sum()) == int(n > 20)
    srv.close()


def test_request_of_one_tile_per_cta_with_scores_that_overflow():
    """The kernel of one CTA per tile (too many candidates for the clusters) where 2^score leaves fp32: it repeats the softmax with exact row
    maxima, as the clusters do (the sharp-softmax test's single launch).  Activations of magnitude A carry about 2^-9 A of rounding error."""
    wl = helpers.MINI["c2"].with_(name="sharp_tiles", R=1, N=2000, L=200, mini_batch=0)
    weights, table = synth.make_weights(wl, zero_bias=False), synth.make_item_table(wl)
    table["E"] = synth.to_bf16_bits(synth.bf16_bits_to_f32(table["E"]) * 32.0)
    rq = synth.make_request(wl, 0)
    rq["S"] = synth.to_bf16_bits(synth.bf16_bits_to_f32(rq["S"]) * 1024.0)
    srv = serving.Server(wl, weights, table)
    st = srv.precompute(1, srv.upload_request(rq, B.USER_PROJECTED))
    ids = synth.IdSampler(wl).request_ids(0)
    got = srv.score_ids(st, ids)[::9]
    want = helpers.make_oracle(wl, weights, M=table["E"].shape[0]).score(table, helpers.projected_request(wl, rq), ids[::9])
    _check(got, want, 1e-2 * max(1.0, float(np.abs(want).max())))
    srv.close()


@pytest.mark.parametrize("H2,L,sigmoid", [(256, 200, 0), (64, 128, 0), (192, 129, 1), (128, 1, 0)])
def test_a_request_in_one_call_or_in_several_gives_the_same_bits(H2, L, sigmoid):
    """A candidate's logit does not depend on how many share its call: clusters of four CTAs (small calls) and one CTA per tile (large ones, and
    batches) sum in the same order, so a request cut into calls on either side of every change is ranked by the bits of the whole."""
    wl = helpers.MINI["c2"].with_(name=f"cut_{H2}_{L}", R=2, N=3000, M=20_000, mini_batch=0, L=L, hidden=(512, H2), emit_sigmoid=sigmoid)
    srv = serving.Server(wl, synth.make_weights(wl, zero_bias=False), synth.make_item_table(wl), path=B.PATH_TENSOR)
    st = srv.precompute(0, srv.upload_request(synth.make_request(wl, 0), B.USER_PROJECTED))
    ids = synth.IdSampler(wl).request_ids(0, 3000)
    whole = srv.score_ids(st, ids)
    assert len(np.unique(whole)) > 1000
    for first in (1, 15, 16, 17, 33, 200, 577, 592, 593, 1000, 1184, 1185, 1728, 1729, 1800):
        assert np.array_equal(srv.score_ids(st, ids[:first]).view(np.uint32), whole[:first].view(np.uint32)), first
        assert np.array_equal(srv.score_ids(st, ids[first:]).view(np.uint32), whole[first:].view(np.uint32)), first
    a, b = srv.score_many([st, st], [ids[:700], ids[700:]])
    assert np.array_equal(np.concatenate([a, b]).view(np.uint32), whole.view(np.uint32))
    srv.close()


def _route(ctx, st, ids, stream):
    """One scoring call on `stream`: the kernels that it took, and its logits."""
    out = torch.empty(ids.numel(), dtype=torch.float32, device="cuda")
    stream.wait_stream(torch.cuda.current_stream())
    ctx.set_kernel_timing(True)
    with torch.cuda.stream(stream):
        ctx.score(st, ids, out)
    names = list(ctx.get_kernel_timing())
    ctx.set_kernel_timing(False)
    torch.cuda.synchronize()
    return names, out.cpu().numpy()


def test_small_requests_on_several_streams_leave_room_for_each_other():
    """Clusters shorten a call by holding most of the machine.  Calls that alternate between streams, of one context or of two, take them only
    where all fit side by side: 1000 candidates on two streams go by the kernel that holds 8 SMs, 200 on two by clusters, 200 on eight
    not; and by clusters again once the calls are on one stream.  The logits are the same bits by any way."""
    wl = helpers.MINI["c2"].with_(name="streams", R=2, N=1000, M=20_000, mini_batch=0, L=200)
    weights, table = synth.make_weights(wl, zero_bias=False), synth.make_item_table(wl)
    srvs = [serving.Server(wl, weights, table, path=B.PATH_TENSOR) for _ in range(2)]
    sts = [s.precompute(0, s.upload_request(synth.make_request(wl, 0), B.USER_PROJECTED)) for s in srvs]
    torch.cuda.synchronize()
    ids = torch.from_numpy(np.ascontiguousarray(synth.IdSampler(wl).request_ids(0, 1000), dtype=np.int32)).cuda()
    streams = [torch.cuda.Stream() for _ in range(8)]

    def go(which, n, stream):
        return _route(srvs[which].ctx, sts[which], ids[:n], streams[stream])

    alone = [go(0, 1000, 0) for _ in range(8)][-1]   # eight calls later nothing of what ran before counts
    assert alone[0] == ["score_split"]
    for two in (0, 1):
        beside = [go(two * (i & 1), 1000, i & 1) for i in range(9)][1:]
        for names, out in beside:
            assert names == ["score_fused"] and np.array_equal(out.view(np.uint32), alone[1].view(np.uint32))
        for i in range(9):
            names, out = go(two * (i & 1), 200, i & 1)
            assert names == ["score_split"] and np.array_equal(out.view(np.uint32), alone[1][:200].view(np.uint32))
    many = [go(0, 200, i) for i in range(8)]
    assert many[-1][0] == ["score_fused"] and np.array_equal(many[-1][1].view(np.uint32), alone[1][:200].view(np.uint32))
    assert [go(0, 1000, 0)[0] for _ in range(8)][-1] == ["score_split"]
    for s in srvs:
        s.close()
