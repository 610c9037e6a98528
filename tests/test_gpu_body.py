"""GPU parity of the one-launch transformer body (small canvases) against the CPU oracle, at the sizes where
its tiling changes: row counts around the 16-row granularity of the token operand, on both sides of 128 rows (two
accumulator pairs or one), few enough for several CTAs to share a row or not, one or two attention items side by side,
K ranges from 1 to 8, ragged tiles."""
import pytest
import torch

from helpers import REL_TOL, compare_stats, oracle_stats_for_rows
from oracle import model_oracle as mo
from paper_2602_11133_b200 import inputs

pytestmark = pytest.mark.gpu

GEOMS = {
    "gqa": inputs.ModelGeometry(2, 256, 4, 2, 64, 320, 1032, 1000, 10000.0),
    "hd128": inputs.ModelGeometry(2, 256, 2, 1, 128, 704, 2048, 2047, 500000.0),
    # wide enough for K ranges of every projection, a ragged last tile of each (3200 + 2 x 640 and 1600 weight rows) and a
    # gate/up projection whose last tile is not full
    "wide": inputs.ModelGeometry(2, 1600, 25, 5, 128, 2368, 1032, 1000, 10000.0),
}


@pytest.fixture(scope="module")
def jot():
    from paper_2602_11133_b200 import jot as binding
    binding._lib()
    return binding


@pytest.mark.parametrize("name,B,P,G", [
    ("gqa", 1, 0, 1),           # one row
    ("hd128", 1, 5, 11),        # 16 rows: one whole granule
    ("hd128", 1, 6, 11),        # 17
    ("wide", 1, 17, 16),        # 33 rows, four CTAs a row
    ("wide", 2, 20, 18),        # 76 rows: one CTA a row
    ("wide", 1, 52, 60),        # 112 rows: the last size with two accumulator pairs; attention items side by side
    ("gqa", 3, 20, 23),         # 129 rows: the first with one
    ("hd128", 2, 40, 32),       # 144 rows: the last size of a wide model
    ("wide", 18, 3, 5),         # 144 rows of 18 short sequences: one key block, items side by side
    ("gqa", 1, 70, 79),         # 149 rows: more rows than CTAs
    ("hd128", 2, 64, 64),       # 256 rows: the last size
])
def test_step_matches_oracle(jot, name, B, P, G):
    g = GEOMS[name]
    w_cpu = inputs.model_weights(g, seed=0)
    L = P + G
    tokens = inputs.partially_masked_canvas(1, B, P, G, g.vocab, g.mask_id, 0.6)
    tokens[:, L - 1] = g.mask_id
    model = jot.Model(g, inputs.weights_to(w_cpu, "cuda"), B, L)
    before = jot.launch_count()
    st = model.denoise_step(tokens.cuda(), P, L)
    assert jot.launch_count() - before == 3                        # body, head, merge
    again = model.denoise_step(tokens.cuda(), P, L)
    rows = [(b, i) for b in range(B) for i in range(P, L) if int(tokens[b, i]) == g.mask_id]
    want = oracle_stats_for_rows(mo.logits(g, w_cpu, tokens, rows=rows), g.mask_id)
    flat = torch.tensor([b * L + i for b, i in rows])
    pick = lambda t: t.cpu().view(-1)[flat].numpy()
    compare_stats(pick(st.top1), pick(st.top2), pick(st.sumexp), pick(st.argmax), want, rel=REL_TOL, gap_from_error=True)
    for a, b in ((st.top1, again.top1), (st.top2, again.top2), (st.sumexp, again.sumexp), (st.argmax, again.argmax)):
        assert torch.equal(a, b)                                   # the order of the sums is fixed
    model.close()


@pytest.mark.parametrize("name,B,P,G,lo,hi", [
    ("gqa", 6, 30, 100, 51, 69),     # 108 rows, items side by side: five key blocks over four warps
    ("wide", 1, 20, 55, 31, 36),     # five rows at an odd position; the last of three key blocks is ragged
    ("hd128", 3, 40, 300, 97, 129),  # eleven key blocks: every warp has one, some two
    ("wide", 2, 3, 20, 3, 23),       # one key block
])
def test_block_pass_matches_oracle(jot, name, B, P, G, lo, hi):
    g = GEOMS[name]
    w_cpu = inputs.model_weights(g, seed=0)
    L = P + G
    canvas0 = inputs.partially_masked_canvas(1, B, P, G, g.vocab, g.mask_id, 0.8)
    canvas0[:, lo:hi] = g.mask_id
    canvas1 = canvas0.clone()
    canvas1[:, lo:hi:2] = inputs.prompt(5, B, len(range(lo, hi, 2)), g.vocab, g.mask_id)
    model = jot.Model(g, inputs.weights_to(w_cpu, "cuda"), B, L)
    model.attach_kv_cache()
    model.denoise_step_cached(canvas0.cuda(), lo, hi, refresh=True)
    st = model.denoise_step_cached(canvas1.cuda(), lo, hi, refresh=False)
    cache = []
    mo.hidden_states(g, w_cpu, canvas0, cache_out=cache)
    h = mo.hidden_states_cached(g, w_cpu, canvas1, cache, lo, hi)
    rows = [(b, i) for b in range(B) for i in range(lo, hi) if int(canvas1[b, i]) == g.mask_id]
    want = oracle_stats_for_rows(mo.lm_head_logits(torch.stack([h[b, i - lo] for b, i in rows]), w_cpu["lm_head"]), g.mask_id)
    flat = torch.tensor([b * L + i for b, i in rows])
    pick = lambda t: t.cpu().view(-1)[flat].numpy()
    compare_stats(pick(st.top1), pick(st.top2), pick(st.sumexp), pick(st.argmax), want, rel=REL_TOL, gap_from_error=True)
    model.close()
