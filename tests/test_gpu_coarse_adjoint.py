"""The coarse levels of the adjoint of recomposition in one block
(coarse_adjoint_kernel): the smallest grids, one to three active dimensions,
short last intervals and sizes on both sides of its shared memory, against the
FP64 oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPES = [(2, 3), (4,), (5, 2), (3, 3, 3), (4, 4, 4), (17, 16, 15), (16, 2, 33), (64, 65), (24, 24, 24), (1500,),
          (2500,), (6001,)]


@pytest.mark.parametrize("shape", SHAPES, ids=str)
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_coarse_adjoint(oracle, shape, dtype):
    from paper_2503_06322_gb300 import hpdr as H
    tol = 1e-5 if dtype == np.float32 else 1e-12     # the parity bar of this path
    g = np.random.default_rng(3).standard_normal(shape).astype(dtype)
    got = H.hpdr_recompose_adjoint(torch.from_numpy(g).cuda()).cpu().numpy().reshape(-1)
    ref = np.asarray(oracle.recompose_adjoint(g.astype(np.float64))).reshape(-1)
    assert np.abs(got - ref).max() <= tol * np.abs(ref).max()
