"""Fixed-rate ZFP at the ends of its number range, where the binary32 scaling
takes two steps or gives way to binary64: subnormal, tiny and huge blocks, wide
ranges inside a block, against the oracle bit for bit."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exponent", [-148, -130, -100, -98, 0, 96, 122, 127])
@pytest.mark.parametrize("shape,rate", [((37, 10, 131), 8), ((33, 70), 6), ((1003,), 24)], ids=str)
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_number_range(oracle, shape, rate, dtype, exponent):
    from paper_2503_06322_gb300 import hpdr as H
    rng = np.random.default_rng(exponent + 200)
    e = 8 * exponent if dtype == np.float64 else exponent
    e = max(e, -1073)
    with np.errstate(under="ignore"):
        x = np.ldexp(rng.random(shape) * 2 - 1, e - rng.integers(0, 60, shape) * rng.integers(0, 2, shape))
        u = x.astype(dtype)
    buf = H.hpdr_zfp_compress(torch.from_numpy(u).cuda(), rate)
    ob = oracle.zfp_compress(u, rate)
    assert np.array_equal(buf.cpu().numpy(), ob)
    got = H.hpdr_zfp_decompress(buf).cpu().numpy()
    assert np.array_equal(got, oracle.zfp_decompress(ob).astype(dtype).reshape(shape))
