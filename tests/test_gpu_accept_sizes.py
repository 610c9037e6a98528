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
