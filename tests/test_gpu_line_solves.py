"""Solves along the contiguous dimension: lines that are and are not a multiple of
eight nodes long, tiles of 32 lines down to few, the lengths at which a tile takes
more shared memory and lines leave it, through decomposition, recomposition and the
adjoint of recomposition (the solution added to, subtracted from and stored), against
the FP64 oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

# the finest level's coarse lines: 8, 9, 16, 33, 128, 129, 500, 504, 1163, 1200, 2049, 2601, 8001
SHAPES = [(40, 60, 15), (40, 60, 16), (36, 61, 31), (33, 34, 64), (5, 67, 255), (9, 31, 257), (3, 70, 998), (3, 45, 1007),
          (33, 2325), (9, 2399), (35, 4097), (5, 5201), (3, 16001)]


@pytest.mark.parametrize("shape", SHAPES, ids=str)
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_line_solves(oracle, shape, dtype):
    from paper_2503_06322_gb300 import hpdr as H
    tol = 1e-5 if dtype == np.float32 else 1e-12     # the parity bar of this path
    u = np.random.default_rng(17).standard_normal(shape).astype(dtype)
    ut = torch.from_numpy(u).cuda()
    ref = np.asarray(oracle.decompose(u.astype(np.float64))).reshape(-1)
    got = H.hpdr_decompose(ut)
    assert np.abs(got.cpu().numpy() - ref).max() <= tol * np.abs(ref).max()
    assert np.abs(H.hpdr_recompose(got, shape).cpu().numpy() - u).max() <= tol * np.abs(u).max()
    ref = np.asarray(oracle.recompose_adjoint(u.astype(np.float64))).reshape(-1)
    assert np.abs(H.hpdr_recompose_adjoint(ut).cpu().numpy() - ref).max() <= tol * np.abs(ref).max()
