"""Whole steps against the CPU oracle at the row counts and layer widths where the cut of the work changes."""
import pytest
import torch

from helpers import REL_TOL, compare_stats, oracle_stats_for_rows
from oracle import model_oracle as mo
from paper_2602_11133_b200 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def jot():
    from paper_2602_11133_b200 import jot as binding
    binding._lib()
    return binding


def check_step(jot, g, B, L):
    w_cpu = inputs.model_weights(g, seed=0)
    P = L // 2 if L > 1 else 0
    tokens = inputs.partially_masked_canvas(1, B, P, L - P, g.vocab, g.mask_id, 0.3)
    tokens[:, L - 1] = g.mask_id
    model = jot.Model(g, inputs.weights_to(w_cpu, "cuda"), B, L)
    st = model.denoise_step(tokens.cuda(), P, L)
    again = model.denoise_step(tokens.cuda(), P, L)
    for a, b in ((st.top1, again.top1), (st.top2, again.top2), (st.sumexp, again.sumexp), (st.argmax, again.argmax)):
        assert torch.equal(a, b)
    rows = [(b, i) for b in range(B) for i in range(P, L) if int(tokens[b, i]) == g.mask_id]
    want = oracle_stats_for_rows(mo.logits(g, w_cpu, tokens, rows=rows), g.mask_id)
    flat = torch.tensor([b * L + i for b, i in rows])
    pick = lambda t: t.cpu().view(-1)[flat].numpy()
    compare_stats(pick(st.top1), pick(st.top2), pick(st.sumexp), pick(st.argmax), want, rel=REL_TOL, gap_from_error=True)
    model.close()


def geometry(d, heads, hd, ff, layers=2):
    return inputs.ModelGeometry(layers, d, heads, heads, hd, ff, 1032, 1000, 10000.0)


# rows of the norm: one, two, three and more vectors per thread
@pytest.mark.parametrize("d,B,L", [(64, 1, 20), (4096, 1, 20), (4160, 1, 20), (8256, 1, 20), (320, 9, 133)])     # ... and more rows than CTAs
def test_norm_widths(jot, d, B, L):
    check_step(jot, geometry(d, 2, 64, 128, layers=1), B, L)


# pair tiles narrower than 256 columns: halves of 112 and of 64 gate columns, O and down in tiles of 240 and less; the last tile and
# the last row block ragged; more row blocks than a band has
@pytest.mark.parametrize("d,ff,B,L", [(256, 1984, 8, 125), (256, 1024, 8, 125), (512, 3968, 4, 130), (4096, 512, 8, 125), (256, 512, 18, 131)])
def test_pair_tile_widths(jot, d, ff, B, L):
    check_step(jot, geometry(d, d // 64, 64, ff, layers=1), B, L)
