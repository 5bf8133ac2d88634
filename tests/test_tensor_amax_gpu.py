"""Both forms of the tensor-maximum kernel (a cluster per matrix; a grid with atomics): one value per matrix, found at the
first, the last and a middle element, at sizes around the line between the forms and around their loop strides."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,rows,cols", [(1, 1, 8), (3, 4097, 128), (1, 4096 * 4, 32), (1, 4096 * 4 + 1, 32), (7, 8200, 128), (8, 8200, 128),
                                             (9, 1023, 64), (2, 70001, 8), (1, 16384, 128), (1, 16385, 128), (4, 11264, 128), (4, 11265, 128)])
def test_maximum_of_every_matrix(batch, rows, cols):
    import paper_2607_24377_b200 as mx
    n = rows * cols
    for where in (0, n // 2, n - 1):
        x = torch.randn(batch, n, device="cuda").clamp_(-6, 6).to(torch.bfloat16)
        peaks = torch.arange(8, 8 + batch, device="cuda", dtype=torch.float32)
        x[:, where] = (peaks * torch.where(torch.arange(batch, device="cuda") % 2 == 0, 1.0, -1.0)).to(torch.bfloat16)
        got = torch.full((batch + 2,), float("nan"), device="cuda")
        mx.tensor_amax(x, got, batch, rows, cols)
        assert torch.equal(got[:batch], peaks) and bool(torch.isnan(got[batch:]).all())
