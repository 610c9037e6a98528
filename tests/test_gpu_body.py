"""GPU parity of the one-launch transformer body (at most 37 rows of a model with large layers) against the CPU oracle, at
the sizes where its tiling changes: row counts around the 16-row granularity of the token operand,
one or two attention items side by side, K ranges, ragged tiles."""
import pytest
import torch

from helpers import REL_TOL, compare_stats, oracle_stats_for_rows
from oracle import model_oracle as mo
from paper_2602_11133_b200 import inputs

pytestmark = pytest.mark.gpu

# layers of at least 96 MB, from which on the body is one launch; ragged last tiles of QKV (3584 and 3072 rows: whole;
# 2624 rows of O and down: not) and of gate/up
GEOMS = {
    "hd128": inputs.ModelGeometry(2, 2624, 20, 4, 128, 5696, 1032, 1000, 10000.0),
    "hd64": inputs.ModelGeometry(1, 2624, 40, 8, 64, 5696, 1032, 1000, 10000.0),
}


@pytest.fixture(scope="module")
def weights():
    made = {}

    def get(name):
        if name not in made:
            cpu = inputs.model_weights(GEOMS[name], seed=0)
            made[name] = (cpu, inputs.weights_to(cpu, "cuda"))
        return made[name]
    return get


@pytest.fixture(scope="module")
def jot():
    from paper_2602_11133_b200 import jot as binding
    binding._lib()
    return binding


@pytest.mark.parametrize("name,B,P,G", [
    ("hd128", 1, 0, 1),         # one row
    ("hd64", 1, 5, 11),         # 16 rows: one whole granule of the token operand
    ("hd128", 1, 6, 11),        # 17
    ("hd128", 1, 10, 22),       # 32 rows
    ("hd64", 7, 2, 3),          # 35 rows of seven short sequences: 280 attention items, side by side
    ("hd128", 1, 17, 20),       # 37 rows: the last size
])
def test_step_matches_oracle(jot, weights, name, B, P, G):
    g = GEOMS[name]
    w_cpu, w_gpu = weights(name)
    L = P + G
    tokens = inputs.partially_masked_canvas(1, B, P, G, g.vocab, g.mask_id, 0.6)
    tokens[:, L - 1] = g.mask_id
    model = jot.Model(g, w_gpu, B, L)
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
    ("hd128", 1, 20, 55, 31, 36),    # five rows at an odd position; the last of three key blocks is ragged
    ("hd64", 1, 40, 300, 97, 129),   # 32 rows, eleven key blocks: every warp has one, some two
    ("hd128", 8, 30, 100, 51, 55),   # 32 rows of 8 sequences, items side by side: five key blocks over four warps
])
def test_block_pass_matches_oracle(jot, weights, name, B, P, G, lo, hi):
    g = GEOMS[name]
    w_cpu, w_gpu = weights(name)
    L = P + G
    canvas0 = inputs.partially_masked_canvas(1, B, P, G, g.vocab, g.mask_id, 0.8)
    canvas0[:, lo:hi] = g.mask_id
    canvas1 = canvas0.clone()
    canvas1[:, lo:hi:2] = inputs.prompt(5, B, len(range(lo, hi, 2)), g.vocab, g.mask_id)
    model = jot.Model(g, w_gpu, B, L)
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
