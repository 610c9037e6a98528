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


# rows of the norm: one, two, three and more vectors per thread; then more rows than CTAs with each of the three instances
@pytest.mark.parametrize("d,B,L", [(64, 1, 20), (4096, 1, 20), (4160, 1, 20), (8256, 1, 20), (320, 9, 133), (4160, 3, 133), (8256, 2, 133)])
def test_norm_widths(jot, d, B, L):
    check_step(jot, geometry(d, 2, 64, 128, layers=1), B, L)


# pair tiles narrower than 256 columns: halves of 112 and of 64 gate columns, O and down in tiles of 240 and less; the last tile and
# the last row block ragged
@pytest.mark.parametrize("d,ff,B,L", [(256, 1984, 8, 125), (256, 1024, 8, 125), (512, 3968, 4, 130), (4096, 512, 8, 125), (256, 512, 18, 131)])
def test_pair_tile_widths(jot, d, ff, B, L):
    check_step(jot, geometry(d, d // 64, 64, ff, layers=1), B, L)


# activations that are walked in bands, an odd number of row blocks, the last band shorter: down (5 and 4 of 9 row-block pairs), then QKV
# and gate/up (six times 8, then 2 of 50)
@pytest.mark.parametrize("d,heads,ff,B,L", [(256, 4, 12032, 15, 140), (2048, 2, 640, 97, 130)])
def test_bands(jot, d, heads, ff, B, L):
    check_step(jot, geometry(d, heads, 64, ff, layers=1), B, L)


# gate/up as two units per pair: a K of fewer blocks than stages, of as many, and more
@pytest.mark.parametrize("d", [64, 128, 192, 320, 576])
@pytest.mark.parametrize("B,L", [(1, 353), (1, 384)])
def test_two_unit_gate_up(jot, d, B, L):
    check_step(jot, geometry(d, d // 64, 64, 12288, layers=1), B, L)


# gate/up dealt over the SMs eight features at a time: 704 (a CTA of 8 each), 9600 (72, the last one ragged), 18944 (128 each), 19200 (two
# units a CTA); the larger passes of 704, 9600 and 19200 in tiles
@pytest.mark.parametrize("ff", [704, 9600, 18944, 19200])
@pytest.mark.parametrize("B,L", [(1, 1), (1, 16), (1, 17), (3, 11), (1, 128), (1, 144), (5, 29), (1, 255), (1, 256)])
def test_small_canvases(jot, ff, B, L):
    check_step(jot, geometry(256, 4, 64, ff), B, L)


# two and three units a CTA, both kinds of accumulators (two up to 128 rows); with 21 k-blocks the rings turn over inside a unit
@pytest.mark.parametrize("d,ff", [(1344, 19200), (256, 38400), (1344, 38400)])
@pytest.mark.parametrize("B,L", [(1, 17), (1, 128), (1, 144)])
def test_several_units_a_cta(jot, d, ff, B, L):
    check_step(jot, geometry(d, 4, 64, ff, layers=1), B, L)


# wide layers of few rows, a ragged last slab of features: four, three and two K ranges of O and down
@pytest.mark.parametrize("d", [1344, 4672, 6464])
@pytest.mark.parametrize("B,L", [(1, 33), (1, 133), (2, 120)])
def test_small_canvases_of_long_sums(jot, d, B, L):
    check_step(jot, geometry(d, 24, 128, 3200, layers=1), B, L)


def statistics(jot, g, weights, tokens, lo):
    model = jot.Model(g, weights, *tokens.shape)
    st = model.denoise_step(tokens, lo, tokens.shape[1])
    model.close()
    return [t[:, lo:] for t in (st.top1, st.top2, st.sumexp, st.argmax)]


def masked_canvas(g, B, L, n_masked):
    tokens = inputs.token_ids(3, "canvas", B * L, g.vocab, g.mask_id, device="cuda").view(B, L)
    tokens[:, L - n_masked:] = g.mask_id
    return tokens


# down adds the same K ranges in the same order with a norm behind it (streams) and as the last layer's (slabs): a second layer that
# adds nothing changes no bit.  (4096 columns have a range more beyond 128 rows.)
@pytest.mark.parametrize("d,heads,hd,ff,L", [(4096, 32, 128, 3072, L) for L in (20, 96, 128)] + [
    (*widths, L) for widths in ((256, 4, 64, 704), (3584, 28, 128, 2048), (4672, 4, 64, 2048), (8192, 4, 64, 1088)) for L in (20, 128, 133, 256)])
def test_same_bits_with_a_norm_behind_and_without(jot, d, heads, hd, ff, L):
    g = geometry(d, heads, hd, ff)
    weights = inputs.model_weights(g, seed=0, device="cuda")
    tokens = masked_canvas(g, 1, L, 16)
    first, second = weights["layers"]
    nothing = dict(second, wo=torch.zeros_like(second["wo"]), w_down=torch.zeros_like(second["w_down"]))
    one = statistics(jot, g, dict(weights, layers=[first]), tokens, L - 16)
    two = statistics(jot, g, dict(weights, layers=[first, nothing]), tokens, L - 16)
    for a, b in zip(one, two):
        assert torch.equal(a, b)


# the norm in the tail of a split projection adds a row's squares in the order of the norm on its own: a sequence gets the same bits
# alone and in a batch, where no projection is split (O and down have one K range that is not zero, so that their sums are the same)
# (20 rows have gate/up as a stream, the others in tiles.)
@pytest.mark.parametrize("d,heads,hd", [(3584, 28, 128), (4096, 32, 128), (5120, 32, 128)])
@pytest.mark.parametrize("B,L", [(9, 100), (45, 20)])
def test_same_bits_of_both_norms(jot, d, heads, hd, B, L):
    g = geometry(d, heads, hd, 4096)
    weights = inputs.model_weights(g, seed=0, device="cuda")
    for layer in weights["layers"]:
        layer["wo"][:, heads * hd // 256 * 64:] = 0
        layer["w_down"][:, g.d_ff // 4:] = 0
    tokens = masked_canvas(g, B, L, 2)
    batch = statistics(jot, g, weights, tokens, L - 2)
    for b in (0, B - 1):
        for x, y in zip(statistics(jot, g, weights, tokens[b:b + 1].contiguous(), L - 2), batch):
            assert torch.equal(x[0], y[b])


# a model keeps what it knows of its weights between passes: passes of other rows in between (other widths of the pair tiles, streams,
# slabs) change no bit
def test_same_bits_whatever_came_before(jot):
    g = geometry(512, 8, 64, 3968)
    weights = inputs.model_weights(g, seed=0, device="cuda")
    shapes = [(8, 200), (1, 200), (5, 130), (8, 200), (8, 125), (1, 40), (5, 130), (3, 200), (8, 125)]
    model = jot.Model(g, weights, 8, 200)
    for B, L in shapes:
        tokens = masked_canvas(g, B, L, 8)
        st = model.denoise_step(tokens, L - 8, L)
        for got, want in zip((st.top1, st.top2, st.sumexp, st.argmax), statistics(jot, g, weights, tokens, L - 8)):
            assert torch.equal(got[:, L - 8:], want)
    model.close()


# gate/up of fewer rows is less work and takes no longer: 257 to 352 rows of the LLaDA-8B widths against 384 (pair tiles of 224 columns
# took 1.07 times as long), 96 to 256 rows of smaller layers against 300 (the stream of weights took up to 1.7 times as long)
@pytest.mark.parametrize("d,heads,hd,ff,fewer,rows", [(4096, 32, 128, 12288, (257, 300, 352), 384), (2048, 16, 128, 5632, (64, 128, 256), 300),
                                                      (2048, 16, 128, 8192, (128, 256), 300), (1024, 16, 64, 2816, (128, 256), 300)])
def test_fewer_rows_take_no_longer(jot, d, heads, hd, ff, fewer, rows):
    g = geometry(d, heads, hd, ff, layers=4 if d < 4096 else 1)
    weights = inputs.model_weights(g, seed=0, device="cuda")

    def gate_up(L):
        model = jot.Model(g, weights, 1, L)
        tokens = torch.full((1, L), 5, dtype=torch.int32, device="cuda")
        best = float("inf")
        for _ in range(8):
            model.profile(True)
            for _ in range(10):
                model.denoise_step(tokens, 0, 0)
            ms, spans = model.profile_read()["gemm_gate_up"]
            best = min(best, ms / spans)
            model.profile(False)
        model.close()
        return best

    full = gate_up(rows)
    for few in fewer:
        assert gate_up(few) <= 1.03 * full, few
