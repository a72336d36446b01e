"""Kernels at the sizes where their tilings change: edges of tiles, ragged
remainders, the smallest inputs and ones larger than a single pass over the
GPU. Each against the oracle or a plain FP64 evaluation, with tolerances that
follow from the arithmetic (stated at each test)."""
import numpy as np
import pytest

import paper_1007_3458_gb300 as q
from oracle import mlp as M
from paper_1007_3458_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch
    assert torch.cuda.is_available()
    return torch


@pytest.mark.parametrize("n", [1, 15, 17, 152 * 16 + 1, 152 * 16 * 8 + 5])
def test_gradient_tiles(torch, n):
    """Guess-network gradient: one row, ragged 16-row tiles, one tile more
    than the CTAs, one tile more than the warps of the whole grid. An entry is
    a sum of products of bf16 operands: a hidden unit near a rounding midpoint
    moves its terms by 2^-8, twice on the way through both layers, so every
    entry stays within 2^-6 of its absolute term sum (FP32 sums far below)."""
    rows = W.mlp_rows_synthetic(n, 14)
    ref = W.mlp_rows_synthetic(4096, 15)
    w = W.mlp_init(5, ref[:, :4], ref[:, 4])
    work = torch.empty(q.qym_mlp_workspace_bytes(), dtype=torch.uint8, device="cuda")
    g = torch.empty(q.QYM_MLP_NW, dtype=torch.float32, device="cuda")
    loss = torch.empty(1, dtype=torch.float32, device="cuda")
    q.qym_mlp_grad_dev(n, torch.from_numpy(w).cuda(), torch.from_numpy(rows).cuda(), g, loss, work)
    L, go, gabs = M.loss_and_grad(w, rows[:, :4], rows[:, 4], emulate=True)
    d = np.abs(g.cpu().numpy().astype(np.float64) - go)
    assert np.all(d <= 2.0 ** -6 * gabs + 1e-7 * np.abs(go).max()), np.max(d / (gabs + 1e-300))
    assert abs(loss.item() - L) <= 1e-4 * L + 1e-7
