"""The acceptance kernel at block lengths around its tiling (warps, 32 to 256 positions side by side, more positions than
threads) and canvases longer than the part it reads ahead, against the CPU oracle, decision by decision."""
import numpy as np
import pytest
import torch

from helpers import oracle_accept_batch
from oracle import jot_oracle as jo
from test_gpu_kernels import random_accept_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def jot():
    from paper_2602_11133_b200 import jot as binding
    binding._lib()
    return binding


@pytest.mark.parametrize("after_exit", [False, True])
@pytest.mark.parametrize("lo,n,L", [(0, 1, 1), (7, 31, 40), (5, 33, 100), (64, 64, 128), (1, 65, 67), (100, 129, 769),
                                    (30, 256, 800), (11, 257, 300), (3, 600, 900)])
def test_accept_freeze_at_block_lengths(jot, lo, n, L, after_exit):
    V, mask_id, B, k = 5000, 4321, 3, 4
    params = jo.JotParams(8.0, 1.0, 0.5, 8)
    tokens, top1, top2, sumexp, argmax = random_accept_case(n * 7 + L, B, L, lo, mask_id, V)
    sumexp[:, lo + n // 2:lo + n] = sumexp[:, lo + n // 2:lo + n // 2 + 1]          # equal sums: the lower position wins
    want, reps = oracle_accept_batch(torch.from_numpy(tokens), top1, top2, sumexp, argmax, params, mask_id, lo, lo + n, k, after_exit)
    d_tok = torch.from_numpy(tokens).cuda()
    st = jot.Stats(*[torch.from_numpy(t).cuda() for t in (top1, top2, sumexp, argmax)])
    n_masked = torch.full((B,), -1, dtype=torch.int32, device="cuda")
    jot.accept_freeze(jot.Params(params.tau_max, params.tau_min, params.gamma, params.D, params.eps, int(after_exit)), mask_id, d_tok,
                      lo, lo + n, k, st, n_masked)
    got = d_tok.cpu()
    for b in range(B):
        if reps[b].near_margin:                                    # a float decision inside the margin may differ
            assert len(reps[b].near_margin) <= 1 + n // 100
            continue
        assert torch.equal(got[b], want[b])
        assert int(n_masked[b]) == int((want[b, lo:lo + n] == mask_id).sum())


@pytest.mark.parametrize("lo,n,L", [(7, 31, 40), (64, 64, 128), (1, 65, 67), (11, 257, 300), (3, 600, 900)])
def test_global_gap_gate_then_schedule_at_block_lengths(jot, lo, n, L):
    """All candidates exit together or none does, and the schedule ranks what is left: nothing, or all of them."""
    V, mask_id, B, k = 5000, 4321, 4, 3
    tokens, top1, top2, sumexp, argmax = random_accept_case(n * 13 + L, B, L, lo, mask_id, V)
    candidate = tokens[:, lo:lo + n] == mask_id
    means = sorted(float((top1 - top2)[b, lo:lo + n][candidate[b]].mean()) for b in range(B))
    thr = max((b - a, (a + b) / 2) for a, b in zip(means, means[1:]))[1]          # in the widest gap between two sequences
    params = jo.JotParams(gate="globalgap", gap_threshold=thr)
    want, reps = oracle_accept_batch(torch.from_numpy(tokens), top1, top2, sumexp, argmax, params, mask_id, lo, lo + n, k, True)
    d_tok = torch.from_numpy(tokens).cuda()
    st = jot.Stats(*[torch.from_numpy(t).cuda() for t in (top1, top2, sumexp, argmax)])
    reason = torch.zeros(B, L, dtype=torch.uint8, device="cuda")
    jot.accept_freeze(jot.Params(schedule_after_exit=1, gate=jot.GATE_GLOBAL_GAP, gap_threshold=thr), mask_id, d_tok, lo, lo + n, k, st,
                      exit_reason=reason)
    assert {len(r.exited) > 0 for r in reps} == {True, False}
    for b in range(B):
        assert not reps[b].near_margin
        assert torch.equal(d_tok.cpu()[b], want[b])
        flags = reason[b].cpu()
        assert (flags & 1).nonzero().flatten().tolist() == reps[b].exited
        assert (flags & 2).nonzero().flatten().tolist() == reps[b].scheduled


@pytest.mark.parametrize("after_exit", [0, 1])
@pytest.mark.parametrize("lo,n,L", [(0, 5, 9), (64, 64, 128), (11, 257, 300), (3, 600, 900)])
def test_sum_that_is_no_number_ranks_first(jot, lo, n, L, after_exit):
    """A position whose sum-exp is not a number never exits early, ranks first in the schedule and changes no other rank: with
    one such position and k = 3 it is chosen besides the three smallest sums."""
    V, mask_id, k = 5000, 4321, 3
    rng = np.random.default_rng(n)
    tokens = np.full((1, L), mask_id, dtype=np.int32)
    tokens[:, :lo] = 1
    top1 = np.full((1, L), 4.0, dtype=np.float32)
    top2 = (top1 - 0.25).astype(np.float32)                        # r = e^0.25: below every threshold
    sumexp = (2.0 + rng.permutation(L) / 8.0).astype(np.float32).reshape(1, L)
    argmax = rng.integers(0, mask_id, size=(1, L)).astype(np.int32)
    at = lo + n - 2
    sumexp[0, at] = np.nan
    order = lo + np.argsort(sumexp[0, lo:lo + n])                  # (not a number sorts last)
    chosen = sorted([at] + order[:3].tolist())
    d_tok = torch.from_numpy(tokens).cuda()
    st = jot.Stats(*[torch.from_numpy(t).cuda() for t in (top1, top2, sumexp, argmax)])
    reason = torch.zeros(1, L, dtype=torch.uint8, device="cuda")
    jot.accept_freeze(jot.Params(60.0, 8.0, 0.5, 8, schedule_after_exit=after_exit), mask_id, d_tok, lo, lo + n, k, st, exit_reason=reason)
    assert (reason[0].cpu() != 0).nonzero().flatten().tolist() == chosen
    want = tokens.copy()
    want[0, chosen] = argmax[0, chosen]
    assert torch.equal(d_tok.cpu(), torch.from_numpy(want))


@pytest.mark.parametrize("after_exit", [False, True])
@pytest.mark.parametrize("k", [1, 40])
@pytest.mark.parametrize("lo,n,L,masked", [(2, 256, 260, 0.1), (0, 257, 257, 0.02), (4, 700, 704, 0.05), (3, 3000, 3010, 0.02)])
def test_few_positions_left_of_a_long_block(jot, lo, n, L, masked, k, after_exit):
    V, mask_id, B = 5000, 4321, 2
    params = jo.JotParams(8.0, 1.0, 0.5, 8)
    tokens, top1, top2, sumexp, argmax = random_accept_case(2 * n + k, B, L, L, mask_id, V)       # all decided
    tokens[:, lo:lo + n][np.random.default_rng(n).random((B, n)) < masked] = mask_id
    sumexp = (np.round(sumexp * 4) / 4).astype(np.float32)                                        # many equal sums
    want, reps = oracle_accept_batch(torch.from_numpy(tokens), top1, top2, sumexp, argmax, params, mask_id, lo, lo + n, k, after_exit)
    d_tok = torch.from_numpy(tokens).cuda()
    st = jot.Stats(*[torch.from_numpy(t).cuda() for t in (top1, top2, sumexp, argmax)])
    jot.accept_freeze(jot.Params(params.tau_max, params.tau_min, params.gamma, params.D, params.eps, int(after_exit)), mask_id, d_tok,
                      lo, lo + n, k, st)
    for b in range(B):
        assert not reps[b].near_margin
        assert torch.equal(d_tok.cpu()[b], want[b])


def test_ranking_costs_what_is_left_not_the_block(jot):
    """8192 positions, 5 % of them masked: a twentieth of the entries, 1/400 of the comparisons; an eighth of the time is allowed."""
    V, L = 5000, 8192

    def time_us(masked):
        gen = torch.Generator(device="cuda").manual_seed(1)
        draw = lambda: torch.rand(1, L, device="cuda", generator=gen)
        tokens = torch.where(draw() < masked, V - 1, 5).to(torch.int32)
        top1 = 4 + draw()
        st = jot.Stats(top1, top1 - 0.1, 2 + 5 * draw(), torch.full_like(tokens, V - 1))          # writes mask_id: nothing changes
        call = lambda: jot.accept_freeze(jot.Params(90.0, 50.0), V - 1, tokens, 0, L, 4, st)
        call()
        begin, end = torch.cuda.Event(True), torch.cuda.Event(True)
        begin.record()
        for _ in range(20):
            call()
        end.record()
        end.synchronize()
        return begin.elapsed_time(end) * 50

    assert time_us(0.05) < time_us(1.0) / 8
