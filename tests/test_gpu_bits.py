"""The decisions of steps whose scores tie, and the bits of the statistics they rest on.

The seeded generator repeats its high-entropy rows in the base and in every
branch. Where all of D_j are such rows, a token and [MASK] have the same score in
exact arithmetic, and how each row's fp32 sums round decides between them: that is
how the rows are cut into pieces, by row count, vocabulary and type. So a change of
the cut changes whole decisions, though every statistic stays within 1e-6. Recorded
on a GB300 (CRC-32 of the arrays' bytes, winners in full).
"""
import zlib

import numpy as np
import pytest
import torch

from paper_2608_11742_gb300 import configs, rps, synth

pytestmark = pytest.mark.gpu

SEED = 89


def crc(t):
    return zlib.crc32(t.detach().contiguous().cpu().view(torch.uint8).numpy().tobytes())


def fill(shape, bf16, mixture, valid=None):
    unit = 8 if bf16 else 4
    t = torch.zeros((*shape[:3], -(-shape[3] // unit) * unit), dtype=torch.bfloat16 if bf16 else torch.float32,
                    device="cuda")[..., :shape[3]]
    synth.device_fill(t, SEED, mixture, valid=valid)
    return t


def step_bits(n, L, V, bf16, P, K, lo, hi, k, low):
    """winner per request, then CRCs of the best slots and of the rows' entropies (base, branches)."""
    pos, cnt = np.full((n, L), -1, np.int32), np.zeros(n, np.int32)
    for q in range(n):
        c = synth.ragged_count(SEED, q, lo, hi)
        pos[q, :c], cnt[q] = synth.masked_positions(SEED, q, L, c), c
    z = fill((n, 1 + P * K, L, V), bf16, (low, 0.3, 0.7 - low))
    e = configs.EXERCISE
    step = rps.Step(n, L, V, configs.Params(k, e.r, e.tau_pivot, e.tau, e.lam, P, K), "cuda", z.dtype)
    step.run(z, torch.from_numpy(pos).cuda(), torch.from_numpy(cnt).cuda())
    assert rps.rps_poll_device_status() == (rps.RPS_OK, 0)
    rows = torch.cat([step.base.H.view(n, L)[q, :cnt[q]] for q in range(n)])
    n_branch = step.piv.n_branch_rows.cpu().tolist()
    branch = torch.cat([step.branch.H.view(n, P * K * L)[q, :n_branch[q]] for q in range(n)])
    return step.commit.winner.cpu().tolist(), crc(step.commit.best_slot), crc(rows), crc(branch)


def row_bits(n, V, bf16, k):
    """CRC of zmax, lse, H and P^max (and mu, htrunc) of n rows."""
    z = fill((1, 1, n, V), bf16, (0.3, 0.3, 0.4))
    out = rps.RowStatsBuf.alloc(n, k, "cuda")
    ws = torch.zeros(rps.rps_workspace_bytes(n, V, k, z.dtype), dtype=torch.uint8, device="cuda")
    rps.rps_score_step(z, None, None, 1, n, configs.Params(k_max=max(k, 1)), out, ws,
                       mask_pos=torch.arange(n, dtype=torch.int32, device="cuda"))
    assert rps.rps_poll_device_status() == (rps.RPS_OK, 0)
    return crc(torch.stack([getattr(out, f) for f in ("zmax", "lse", "H", "pmax") + (("mu", "htrunc") if k else ())]))


# (requests, length, vocabulary, bf16, pivots, tokens, masked positions from, to, k, share of one-spike rows)
STEPS = {
    (18, 384, 2601, False, 3, 4, 2, 38, 16, 0.3): ([9, 4, -1, 2, 4, 8, -3, 7, -1, 4, 9, 0, 8, 4, 9, 9, 8, 0],
        3919067997, 2853018594, 1226260874),
    (8, 48, 28187, True, 2, 3, 1, 6, 10, 0.4): ([-3, -1, 0, -3, -1, -3, -3, -3], 3506941406, 1948005585,
        3233065839),
    (10, 48, 13992, False, 8, 2, 1, 24, 10, 0.4): ([1, -1, 6, 1, 11, 2, 14, 3, 6, 12], 708085661, 2139700097,
        2299486943),
    (24, 64, 17524, True, 8, 2, 6, 6, 32, 0.3): ([0, 6, 1, 0, 3, 2, 3, 5, 2, 6, -1, 0, 2, 5, 0, -1, -1, -1, 4, -1,
        -1, 0, 4, 1], 169879390, 1292338567, 1747967199),
    (32, 64, 3107, True, 2, 3, 2, 32, 10, 0.5): ([0, 3, 2, 1, 3, -3, -1, 5, 1, 1, 3, 0, 0, 3, 0, 3, 3, 5, 0, 0, 5,
        0, 1, 0, 1, 4, -3, 0, -1, 4, 3, -1], 146997862, 1291333593, 1389662555),
    (20, 512, 7718, True, 3, 4, 1, 4, 10, 0.3): ([-1, 1, -1, 0, 4, -3, -3, 5, -1, -3, 0, -3, -1, -1, -1, -3, 2,
        -1, 4, 2], 2332912712, 3364910580, 3545431306),
    (22, 48, 69209, True, 8, 2, 1, 4, 10, 0.5): ([-3, 3, -3, 2, -1, -3, -3, -1, -1, -3, -1, -3, 0, -1, -3, -3, -1,
        -1, 2, -3, -3, 2], 3814770588, 4107623121, 3547378359),
    (40, 32, 16000, True, 4, 2, 2, 8, 10, 0.4): ([0, 2, 4, 6, -1, -1, 0, -1, -1, 0, 1, 0, 4, 0, 2, 1, 2, -1, 4,
        -3, 4, -1, 2, -1, 5, 1, -1, 5, -1, 4, -1, 7, 2, -1, -1, -1, 1, 2, 5, 0], 2117692420, 1594056753,
        972557138),
}

# (rows, vocabulary, bf16, k)
ROWS = {
    (1, 1, False, 0): 3121671225,
    (1, 1, False, 1): 3107840523,
    (3, 1023, True, 0): 4144583016,
    (3, 1023, True, 10): 1142720386,
    (5, 1025, True, 0): 3559352444,
    (5, 1025, True, 10): 1096579593,
    (9, 3447, True, 0): 2859395386,
    (9, 3447, True, 10): 1971950358,
    (32, 4096, False, 0): 2659262144,
    (32, 4096, False, 10): 2145627999,
    (7, 15360, False, 0): 1377371446,
    (7, 15360, False, 10): 2123555553,
    (32, 126464, True, 0): 586479677,
    (32, 126464, True, 10): 68425984,
    (141, 33000, True, 0): 1353839718,
    (141, 33000, True, 10): 2770979728,
    (142, 33000, True, 0): 2080772372,
    (142, 33000, True, 10): 3921535748,
    (163, 33000, True, 0): 3477209619,
    (163, 33000, True, 10): 4210773603,
    (700, 9000, False, 0): 2150557913,
    (700, 9000, False, 10): 1811668409,
    (1000, 9807, True, 0): 3607258086,
    (1000, 9807, True, 10): 3072230727,
    (1000, 45000, True, 0): 986291098,
    (1000, 45000, True, 10): 3279186518,
    (256, 126464, True, 0): 2351143094,
    (256, 126464, True, 10): 1554317811,
    (4000, 9807, True, 0): 1662334953,
    (4000, 9807, True, 10): 2170839794,
    (5000, 2050, False, 0): 33037227,
    (5000, 2050, False, 10): 4066566733,
}


@pytest.mark.parametrize("case", STEPS, ids=str)
def test_tied_decisions(case):
    assert step_bits(*case) == STEPS[case]


@pytest.mark.parametrize("case", ROWS, ids=str)
def test_row_bits(case):
    assert row_bits(*case) == ROWS[case]
