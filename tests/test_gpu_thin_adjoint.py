"""Adjoints on grids around the widths at which the prolongation's warps change from
eight to 32 columns, and with rows that end inside a warp, against the FP64 oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPES = [(70, 61, 3), (70, 67, 14), (66, 65, 16), (40, 70, 65), (38, 41, 125), (34, 37, 130), (33, 39, 145), (31, 36, 190),
          (900, 13), (5000, 5), (300, 129)]


@pytest.mark.parametrize("shape", SHAPES, ids=str)
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_thin_adjoints(oracle, shape, dtype):
    from paper_2503_06322_gb300 import hpdr as H
    tol = 1e-5 if dtype == np.float32 else 1e-12     # the parity bar of this path
    g = np.random.default_rng(5).standard_normal(shape).astype(dtype)
    gt = torch.from_numpy(g).cuda()
    ref = np.asarray(oracle.recompose_adjoint(g.astype(np.float64))).reshape(-1)
    got = H.hpdr_recompose_adjoint(gt).cpu().numpy()
    assert np.abs(got - ref).max() <= tol * np.abs(ref).max()
    ref = np.asarray(oracle.decompose_adjoint(g.astype(np.float64).reshape(-1), shape)).reshape(-1)
    got = H.hpdr_decompose_adjoint(gt.view(-1), shape).cpu().numpy().reshape(-1)
    assert np.abs(got - ref).max() <= tol * np.abs(ref).max()
