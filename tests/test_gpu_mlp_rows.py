"""Training gradients at the row counts where the kernel's split changes: one row, a CTA's
first row past a full one, both sides of the 32-, 64- and 96-row variants (152 CTAs of so many
rows), and several passes per CTA.

Tolerance: a gradient is a sum of B terms of at most a few hundred FP32 roundings each way
(rows of a CTA, CTAs, the inner sums of 64), about sqrt(400) 2^-24 = 1.2e-6 of the sum of the
terms' magnitudes; targets well off the outputs keep that sum within ten times the largest
gradient.  Rows with a unit so near zero that FP32 may put it on the other side are masked."""
import numpy as np
import pytest

from oracle import mlp as M
from paper_2401_07965_gb300 import pa

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 33, 152 * 32, 152 * 32 + 1, 152 * 64 + 1, 152 * 96, 152 * 96 + 1])
def test_gradients_at_split_edges(B):
    import torch
    rng = np.random.default_rng(B)
    w = rng.normal(0, 0.3, M.NPARAM).astype(np.float32)
    X = rng.normal(0, 1, (B, M.IN)).astype(np.float32)
    Yt = rng.normal(4, 1, (B, M.OUT)).astype(np.float32)
    mask = (rng.random((B, M.OUT)) > 0.25).astype(np.float32)
    wb = M.bf16_round(w).astype(np.float64)
    z1, _, z2, _ = M.forward64(wb, X)[1]
    mask[np.minimum(np.abs(z1).min(1), np.abs(z2).min(1)) < 2e-5] = 0
    g64, l64 = M.grads64(wb, X.astype(np.float64), Yt.astype(np.float64), mask.astype(np.float64))
    wd, Xd, Yd, Md = (torch.from_numpy(a).cuda() for a in (w, X, Yt, mask))
    g = torch.full((M.NPARAM,), 7.0, device="cuda")
    loss = torch.zeros(1, device="cuda")
    scratch = torch.empty(pa.pa_mlp_scratch_bytes(B), dtype=torch.uint8, device="cuda")
    pa.pa_mlp_gradients(wd.data_ptr(), Xd.data_ptr(), Yd.data_ptr(), Md.data_ptr(), B,
                        g.data_ptr(), loss.data_ptr(), scratch.data_ptr(), scratch.numel(),
                        torch.cuda.current_stream().cuda_stream)
    gd = g.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(gd - g64) <= 2e-5 * np.max(np.abs(g64)) + 1e-4 * np.abs(g64))
    assert abs(loss.item() - l64) <= 1e-5 * l64
