"""Codes of the level kernels where their quantizers change paths: half-bin
points and their neighbours, the edge of the dictionary, escapes, alphabets inside and beyond the shared histogram's window."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [256, 8192, 32768])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("shape", [(38, 65, 129), (257, 130)], ids=str)
def test_level_codes(oracle, shape, dtype, D):
    from paper_2503_06322_gb300 import hpdr as H
    tau, peak = 0.37, 8e3 if dtype == np.float32 else 3e6   # binary32 bounds leave no wider codes
    rng = np.random.default_rng(D)
    q = oracle.bins(shape, tau, peak, 2.0 ** -24 if dtype == np.float32 else 2.0 ** -53)[-1]
    new = np.zeros(shape, bool)                      # zero at the kept nodes: coefficients are the values
    for k, m in enumerate(shape):
        odd = np.arange(m) % 2 == 1
        odd[-1] = False
        new |= odd.reshape([-1 if i == k else 1 for i in range(len(shape))])
    n = int(new.sum())
    top = np.array([3, D // 2, 3 * D, peak / q])[rng.integers(0, 4, n)]
    t = (((rng.random(n) * 2 - 1) * top).astype(np.int64) + 0.5) * q
    edge = rng.integers(0, 8, n) == 0
    t[edge] = (np.array([-1, 1])[rng.integers(0, 2, n)] * (D // 2 - rng.integers(0, 2, n) - 0.5) * q)[edge]
    t = np.clip(t, -peak, peak).astype(dtype)
    step = rng.integers(-1, 2, n)
    t = np.where(step == 0, t, np.nextafter(t, np.where(step > 0, np.inf, -np.inf).astype(dtype)))
    t[0] = peak
    u = np.zeros(shape, dtype)
    u[new] = np.clip(t, -peak, peak)
    ut = torch.from_numpy(u).cuda()
    h = oracle.parse_header(H.hpdr_compress(ut, tau, tol_kind=H.ABS, dict_size=D).cpu().numpy())
    sym, esc = oracle.decode(h["words"], h["chunk"], h["N"], h["K"], h["lengths"], esc_width=h["esc_width"])
    coef = H.hpdr_decompose(ut).cpu().numpy().astype(np.float64)
    assert np.array_equal(coef[-n:], u[new].astype(np.float64))
    ref_sym, ref_idx, ref_k = oracle.quantize(coef, shape, h["q"], D=D, precision=64)
    assert np.array_equal(sym, ref_sym)
    assert np.array_equal(esc, ref_k)
    assert np.abs(ref_k).max() > D
