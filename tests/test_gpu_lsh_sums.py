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


def _run(base, blocks, Ls, sizes, one_by_one=(), **kw):
    wl = helpers.MINI[base].with_(name=f"lsh_sums_{base}_{blocks}", R=len(Ls), N=max(sizes), L=max(Ls), mini_batch=0, blocks=blocks, **kw)
    weights, table = synth.make_weights(wl, zero_bias=False), None
    table = synth.make_item_table(wl)
    srv = serving.Server(wl, weights, table, path=B.PATH_TENSOR, max_batch_candidates=sum(sizes))
    oracle = helpers.make_oracle(wl, weights, M=table["E"].shape[0])
    sampler = synth.IdSampler(wl)
    states, ids, want = [], [], []
    for r, (L, n) in enumerate(zip(Ls, sizes)):
        rq = synth.make_request(wl, r, L=L)
        states.append(srv.precompute(r, srv.upload_request(rq, B.USER_PROJECTED)))
        ids.append(sampler.request_ids(r, n))
        want.append(oracle.score(table, helpers.projected_request(wl, rq), ids[-1]))
    outs = srv.score_many(states, ids)
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


# One long sequence makes the launch one of many key blocks, which is what takes LSH-DIN to the sums; the others are at the edges.
@pytest.mark.parametrize("base,blocks", [("c2", synth.BLK_CROSS | LSH), ("c2", helpers.ALL_BLOCKS), ("c2", synth.BLK_CROSS | synth.BLK_LSH_DIN),
                                         ("c5", synth.BLK_CROSS | LSH), ("c5", synth.BLK_ATT | synth.BLK_CROSS | LSH)])
def test_sequences_at_the_edges_of_blocks_and_units(base, blocks):
    """Key blocks and units of 128 (64 for the pieces at d = 256), up to eight CTAs per request: lengths on either side of each, requests of
    one candidate and of a whole number of tiles, scored together and, a few, alone (the pass over the pairs)."""
    Ls = [1, 63, 65, 127, 128, 129, 255, 256, 257, 385, 640, 1025, 40_001]
    sizes = [1, 127, 128, 129, 33, 300, 64, 31, 256, 1, 130, 700, 2]
    _run(base, blocks, Ls, sizes, one_by_one=(9, 10, 11))


def test_pieces_of_long_sequences():
    """Fewer tiles than SMs: SimTier's counts in pieces of the keys; one tile over a sequence that a counter's lower digits do not hold."""
    _run("c2", synth.BLK_CROSS | LSH, [9001, 4096], [5300, 128], one_by_one=(1,))
    _run("c2", synth.BLK_CROSS | synth.BLK_SIMTIER, [70_000], [3])
    _run("c5", synth.BLK_CROSS | synth.BLK_SIMTIER, [3001], [100])


@pytest.mark.parametrize("base,L", [("c2", 2600), ("c5", 4200)])
def test_more_requests_than_sms(base, L):
    """One CTA per request and column half."""
    n = 160
    _run(base, synth.BLK_CROSS | LSH, [L] + [40 + r for r in range(n - 1)], [3 + r % 5 for r in range(n)], one_by_one=(0,))


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_rows_that_are_not_finite(value):
    """A sequence row with one infinite or missing value: the scores are what the pass over the pairs makes of it."""
    outs = []
    for long in (False, True):
        Ls = [300, 40_001] if long else [300]
        wl = helpers.MINI["c2"].with_(name="lsh_sums_inf", R=2, N=1400, L=max(Ls), mini_batch=0, blocks=synth.BLK_CROSS | LSH)
        table = synth.make_item_table(wl)
        srv = serving.Server(wl, synth.make_weights(wl, zero_bias=False), table, path=B.PATH_TENSOR, max_batch_candidates=3000)
        rqs = [synth.make_request(wl, r, L=L) for r, L in enumerate(Ls)]
        up = [srv.upload_request(rq, B.USER_PROJECTED) for rq in rqs]
        seq = up[0]["seq"]
        seq[17, 5] = float(value)
        states = [srv.precompute(r, u) for r, u in enumerate(up)]
        ids = synth.IdSampler(wl).request_ids(0, 1300)
        outs.append(srv.score_many(states, [ids, ids[:1]][:len(Ls)])[0])
        srv.close()
    assert np.allclose(outs[0], outs[1], rtol=0, atol=2e-3, equal_nan=True)
