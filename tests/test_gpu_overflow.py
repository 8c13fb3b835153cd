"""Fields so large that their coefficients overflow, at bounds so loose that the bins
do too: the code of infinity times zero is not a number and the call is refused, in
the level kernels and in the coarse block."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(33,), (5000,), (129, 65), (40, 41, 42)], ids=str)
@pytest.mark.parametrize("tol", [1.0, 1e3, 1e10])
def test_overflowed_codes_are_refused(shape, tol):
    from paper_2503_06322_gb300 import hpdr as H
    u = torch.full(shape, 1.7e308, dtype=torch.float64, device="cuda")
    u.view(-1)[1::2] = -1.7e308
    assert not torch.isfinite(H.hpdr_decompose(u)).all()
    with pytest.raises(H.HpdrError) as e:
        H.hpdr_compress(u, tol)
    assert e.value.status == -1
