"""Rank-predictor gradient at the edges of its sample tiles (run with -m gpu): one
sample, one short of, exactly and one above a tile of 32, several tiles per CTA.
Against the FP64 oracle, 1e-5 of the largest gradient entry (FP32 sums; as
tests/test_gpu_mlp.py)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 32, 33, 20001])
def test_grad_sizes(orc, n):
    import torch
    import paper_2505_00715_gb300 as td
    rng = np.random.default_rng(n)
    P = (rng.standard_normal(5648) * 0.3).astype(np.float32)
    x = rng.standard_normal((n, 6)).astype(np.float32)
    lab = rng.integers(0, 16, n).astype(np.int32)
    M = td.Model(td.Context(0))
    M.set_params(P)
    loss, g = M.loss_grad(torch.as_tensor(x, device="cuda"), torch.as_tensor(lab, device="cuda"))
    lo, go = orc.mlp_loss_grad(P.astype(np.float64), x.astype(np.float64), lab)
    assert abs(loss.item() - lo) <= 1e-5 * abs(lo)
    assert np.max(np.abs(g.cpu().numpy() - go)) <= 1e-5 * np.max(np.abs(go))
