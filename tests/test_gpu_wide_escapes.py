"""Binary32 fields at bounds just above the precision floor, whose bins are so
small that codes need more than 32 bits: the payloads that do not fit a word, in
the level kernels and in the coarse block, many of them and few, against the
oracle's codes and values."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [256, 8192])
@pytest.mark.parametrize("above", [1e-2, 1e-3, 1e-6])      # about 30, 33 and 43 bits
@pytest.mark.parametrize("shape,spikes", [((38, 65, 129), 0), ((17, 16, 15), 0), ((1025, 1030), 3)], ids=str)
def test_wide_escapes(oracle, shape, spikes, above, D):
    from paper_2503_06322_gb300 import hpdr as H
    rng = np.random.default_rng(11)
    if spikes:      # few escapes: the rest of the field is zero
        u = np.zeros(shape, np.float32)
        u[tuple(rng.integers(0, n, spikes) for n in shape)] = rng.standard_normal(spikes)
    else:
        u = (rng.random(shape) * 2 - 1).astype(np.float32)
    levels = len(oracle.bins(shape, 1.0, 0.0, 0.0))
    tau = 32.0 * levels * 2.0 ** -24 * float(np.abs(u).max()) * (1.0 + above)
    ut = torch.from_numpy(u).cuda()
    out = torch.empty(24 * u.size + (1 << 16), dtype=torch.uint8, device="cuda")
    buf = H.hpdr_compress(ut, tau, tol_kind=H.ABS, dict_size=D, out=out)
    h = oracle.parse_header(buf.cpu().numpy())
    sym, esc = oracle.decode(h["words"], h["chunk"], h["N"], h["K"], h["lengths"], esc_width=h["esc_width"])
    assert above > 1e-6 or h["esc_width"] > 32
    assert above < 1e-2 or h["esc_width"] <= 32
    assert (len(esc) * 16 < u.size) == bool(spikes)
    coef = H.hpdr_decompose(ut).cpu().numpy().astype(np.float64)
    ref_sym, ref_idx, ref_k = oracle.quantize(coef, shape, h["q"], D=D, precision=64)
    assert np.array_equal(sym, ref_sym)
    assert np.array_equal(esc, ref_k)
    got = H.hpdr_decompress(buf).cpu().numpy().astype(np.float64)
    ref = oracle.decompress(buf.cpu().numpy())
    assert np.abs(got - ref).max() <= 1e-5 * np.abs(ref).max()     # the parity bar of this path in binary32
    assert np.abs(got - u).max() <= tau
