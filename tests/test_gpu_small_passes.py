"""Passes of few rows through a model with large layers, where the weights' stream is all there is: parity with the CPU
oracle at row counts around the 16-row granularity of the token operand, K ranges and ragged tiles; the same bits while
kernels are timed; no waiting for what other streams run."""
import pytest
import torch

from helpers import REL_TOL, compare_stats, oracle_stats_for_rows
from oracle import model_oracle as mo
from paper_2602_11133_b200 import inputs

pytestmark = pytest.mark.gpu

# layers of at least 96 MB; whole tiles of QKV (3584 and 3072 rows), ragged last ones of O and down (2624) and of gate/up
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
    ("hd64", 7, 2, 3),          # 35 rows of seven short sequences
    ("hd128", 1, 17, 20),       # 37
])
def test_step_matches_oracle(jot, weights, name, B, P, G):
    g = GEOMS[name]
    w_cpu, w_gpu = weights(name)
    L = P + G
    tokens = inputs.partially_masked_canvas(1, B, P, G, g.vocab, g.mask_id, 0.6)
    tokens[:, L - 1] = g.mask_id
    model = jot.Model(g, w_gpu, B, L)
    st = model.denoise_step(tokens.cuda(), P, L)
    again = model.denoise_step(tokens.cuda(), P, L)
    model.profile(True)
    timed = model.denoise_step(tokens.cuda(), P, L)                # timing changes no result
    model.profile(False)
    rows = [(b, i) for b in range(B) for i in range(P, L) if int(tokens[b, i]) == g.mask_id]
    want = oracle_stats_for_rows(mo.logits(g, w_cpu, tokens, rows=rows), g.mask_id)
    flat = torch.tensor([b * L + i for b, i in rows])
    pick = lambda t: t.cpu().view(-1)[flat].numpy()
    compare_stats(pick(st.top1), pick(st.top2), pick(st.sumexp), pick(st.argmax), want, rel=REL_TOL, gap_from_error=True)
    for other in (again, timed):
        for a, b in ((st.top1, other.top1), (st.top2, other.top2), (st.sumexp, other.sumexp), (st.argmax, other.argmax)):
            assert torch.equal(a, b)                               # the order of the sums is fixed
    model.close()


@pytest.mark.parametrize("name,B,P,G,lo,hi", [
    ("hd128", 1, 20, 55, 31, 36),    # five rows at an odd position; the last of three key blocks is ragged
    ("hd64", 1, 40, 300, 97, 129),   # 32 rows, eleven blocks of 32 keys
    ("hd128", 8, 30, 100, 51, 55),   # 32 rows of 8 sequences
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


def test_pass_does_not_wait_for_other_streams(jot, weights):
    """A one-thread kernel that another stream keeps on one SM for some 50 ms holds up neither a full pass nor a block pass
    (well below 2 ms each)."""
    g = GEOMS["hd128"]
    model = jot.Model(g, weights("hd128")[1], 1, 75)
    model.attach_kv_cache()
    canvas = inputs.partially_masked_canvas(1, 1, 20, 55, g.vocab, g.mask_id, 0.8)
    canvas[:, 31:36] = g.mask_id
    canvas, short = canvas.cuda(), canvas[:, 20:52].cuda()
    model.denoise_step_cached(canvas, 31, 36, refresh=True)
    calls = (lambda: model.denoise_step(short, 11, 16), lambda: model.denoise_step_cached(canvas, 31, 36, refresh=False))
    alone = [call() for call in calls]
    side, ended = torch.cuda.Stream(), torch.cuda.Event()
    for call, want in zip(calls, alone):
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            torch.cuda._sleep(100_000_000)
            ended.record()
        got = call()                                               # returns when its own stream is done
        assert not ended.query()
        torch.cuda.synchronize()
        for a, b in ((got.top1, want.top1), (got.top2, want.top2), (got.sumexp, want.sumexp), (got.argmax, want.argmax)):
            assert torch.equal(a, b)
    model.close()
