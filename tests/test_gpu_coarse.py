"""The coarse levels in one block (coarse_kernel): its forms (tables and stream
staged in shared memory or read in global memory, one to three active
dimensions, short last intervals, the smallest grids) against the FP64 oracle,
and the binary32 decision of its quantizer at the points where only binary64
can decide."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

# 1-D grids above about 2000 nodes keep their tables in global memory
SHAPES = [(2, 3), (4,), (5, 2), (3, 3, 3), (4, 4, 4), (17, 16, 15), (16, 2, 33), (64, 65), (1500,), (2500,), (6001,)]


@pytest.mark.parametrize("shape", SHAPES, ids=str)
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_coarse_levels(oracle, shape, dtype):
    from paper_2503_06322_gb300 import hpdr as H
    tol = 1e-5 if dtype == np.float32 else 1e-12     # the parity bar of this path
    u = np.random.default_rng(7).standard_normal(shape).astype(dtype)
    ut = torch.from_numpy(u).cuda()
    ref = oracle.decompose(u.astype(np.float64))
    got = H.hpdr_decompose(ut)
    assert np.abs(got.cpu().numpy() - ref).max() <= tol * np.abs(ref).max()
    back = H.hpdr_recompose(got, shape).cpu().numpy()
    assert np.abs(back - u).max() <= tol * np.abs(u).max()
    buf = H.hpdr_compress(ut, 1e-3)
    rec = H.hpdr_decompress(buf).cpu().numpy().astype(np.float64)
    assert np.abs(rec - u).max() <= 1e-3 * np.abs(u).max()
    orec = oracle.decompress(buf.cpu().numpy())
    assert np.abs(rec - orec).max() <= tol * np.abs(u).max()


@pytest.mark.parametrize("n", [33, 1025, 4097])
def test_half_bin_decisions(oracle, n):
    """Finest coefficients placed on the binary32 neighbours of (k + 1/2) q:
    every code is the binary64 decision's."""
    from paper_2503_06322_gb300 import hpdr as H
    tau = 0.37
    rng = np.random.default_rng(n)
    u = np.zeros(n, np.float32)
    u[1] = 3000.0                                    # the largest magnitude, fixed
    q = oracle.bins((n,), tau, 3000.0, 2.0 ** -24)[-1]
    k = rng.integers(-1000, 1000, size=u[3::2].size)
    t = ((k + 0.5) * q).astype(np.float32)
    step = rng.integers(-1, 2, size=t.size)
    u[3::2] = np.where(step == 0, t, np.nextafter(t, np.where(step > 0, np.inf, -np.inf).astype(np.float32)))
    buf = H.hpdr_compress(torch.from_numpy(u).cuda(), tau, tol_kind=H.ABS).cpu().numpy()
    h = oracle.parse_header(buf)
    sym, esc = oracle.decode(h["words"], h["chunk"], h["N"], h["K"], h["lengths"], esc_width=h["esc_width"])
    coef = H.hpdr_decompose(torch.from_numpy(u).cuda()).cpu().numpy().astype(np.float64)
    assert np.array_equal(coef[-u[1::2].size:], u[1::2].astype(np.float64))
    ref_sym, ref_idx, ref_k = oracle.quantize(coef, (n,), h["q"], D=8192, precision=64)
    assert np.array_equal(sym, ref_sym)
    assert np.array_equal(esc, ref_k)
