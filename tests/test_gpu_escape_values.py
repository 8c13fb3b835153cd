"""Escaped codes back to values: codes that fit 24 bits, 32 bits and neither, in
the level kernels and in the coarse block, against the FP64 oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,peak", [(np.float32, 8e3), (np.float64, 8e3), (np.float64, 3e6), (np.float64, 1e11)])
@pytest.mark.parametrize("shape", [(38, 65, 129), (17, 16, 15)], ids=str)
def test_escaped_codes_decode(oracle, shape, dtype, peak):
    from paper_2503_06322_gb300 import hpdr as H
    tol = 1e-5 if dtype == np.float32 else 1e-12     # the parity bar of this path
    u = ((np.random.default_rng(9).random(shape) * 2 - 1) * peak).astype(dtype)
    out = torch.empty(16 * u.size + (1 << 16), dtype=torch.uint8, device="cuda")   # the widest codes outgrow the field
    buf = H.hpdr_compress(torch.from_numpy(u).cuda(), 0.37, tol_kind=H.ABS, dict_size=256, out=out)
    got = H.hpdr_decompress(buf).cpu().numpy().astype(np.float64)
    ref = oracle.decompress(buf.cpu().numpy())
    assert np.abs(got - ref).max() <= tol * np.abs(ref).max()
    assert np.abs(got - u).max() <= 0.37
