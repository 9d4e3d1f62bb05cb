"""The row statistics at the edges of the rows' cut into pieces: rows shorter than
one ring chunk, one chunk, one more element; few rows (a warp per part of a row,
spread over the blocks) and the row counts around which the cut changes form.
Against the oracle, in both modes."""
import numpy as np
import pytest
import torch

from gpu_harness import compare_stats, padded_tensor, stats_np
from oracle import default as oracle_default
from paper_2608_11742_gb300 import configs, rps, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,V,bf16", [
    (1, 1, False),         # one piece of one value
    (3, 1023, True),       # a whole chunk's units less one value, in pieces of five units across rows
    (2, 1024, True),       # exactly one chunk
    (5, 1025, True),       # one value more
    (7, 512 * 30, False),  # 30 pieces of one chunk
    (1, 40001, True),      # 30 pieces, the last one short and ragged
    (162, 33000, True),    # 30 pieces a row, none across rows
    (163, 33000, True),    # 29 a row
    (700, 9000, False),    # 6 pieces a row would idle more than an eighth of the warps: the even cut, across rows
    (1000, 45000, True),   # so would 4 long ones
])
@pytest.mark.parametrize("k", [0, 10])
def test_cut(n, V, bf16, k):
    rng = np.random.default_rng(n + V)
    z = rng.standard_normal((1, 1, n, V)).astype(np.float32)
    z[0, 0, np.arange(n), rng.integers(0, V, n)] += rng.uniform(0, 12, n).astype(np.float32)
    host = synth.bf16_round(z) if bf16 else z
    t = padded_tensor(host)
    k = min(k, V)
    out = rps.RowStatsBuf.alloc(n, k, "cuda")
    ws = torch.zeros(rps.rps_workspace_bytes(n, V, k, t.dtype), dtype=torch.uint8, device="cuda")
    pos = torch.arange(n, dtype=torch.int32, device="cuda")
    prm = configs.Params(k_max=max(k, 1))
    for _ in range(2):  # the second call finds the tickets the first one left
        rps.rps_score_step(t, None, None, 1, n, prm, out, ws, mask_pos=pos)
    assert rps.rps_poll_device_status() == (rps.RPS_OK, 0)
    compare_stats(stats_np(out), oracle_default().row_stats(host[0, 0], k), np.arange(n), k, f"{n} x {V}")


@pytest.mark.parametrize("V", [40, 100, 3447, 7680, 7684, 32003])  # few chunks up to V 8,188; a cell a lane from 128
@pytest.mark.parametrize("k", [10, 16, 17, 31, 32])
@pytest.mark.parametrize("kind", ["spread", "equal", "few"])
def test_lists(kind, k, V):
    """The bound of the top-k search (one or two maxima per lane, over vectors of
    cells or over the cells of short rows): spread rows, rows of equal logits, and
    rows of fewer finite logits than k."""
    rng = np.random.default_rng(k + V)
    n = 9
    z = np.zeros((1, 1, n, V), np.float32)
    if kind == "spread":
        z[:] = rng.standard_normal(z.shape)
    elif kind == "few":
        z[:] = -np.inf
        z[0, 0, :, rng.choice(V, k - 3, replace=False)] = rng.standard_normal((k - 3, n)).astype(np.float32)
    t = padded_tensor(z)
    out = rps.RowStatsBuf.alloc(n, k, "cuda")
    ws = torch.zeros(rps.rps_workspace_bytes(n, V, k, t.dtype), dtype=torch.uint8, device="cuda")
    rps.rps_score_step(t, None, None, 1, n, configs.Params(k_max=k), out, ws,
                       mask_pos=torch.arange(n, dtype=torch.int32, device="cuda"))
    assert rps.rps_poll_device_status() == (rps.RPS_OK, 0)
    compare_stats(stats_np(out), oracle_default().row_stats(z[0, 0], k), np.arange(n), k, f"{kind} k={k}")
