"""The rotations of the complex64 Jacobi SVD keep the norm of a matrix in the mean."""
import pytest

pytestmark = pytest.mark.gpu


# The thousands of rotations of an SVD round each value by about 1e-7, to either side: the mean
# over a batch has a standard error of 5e-10.  A sixteenth of the unit roundoff, 3.7e-9, leaves
# seven of them; a cosine that rounds more often up than down shows as 1e-8 and more.
@pytest.mark.parametrize("batch,rows,cols", [(2000, 64, 48), (800, 128, 100), (600, 200, 200)])
def test_norms_neither_grow_nor_shrink(batch, rows, cols):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_02667_gb300 import ptebd
    gen = torch.Generator(device="cuda").manual_seed(7)
    a = torch.view_as_complex(torch.randn((batch, rows, cols, 2), generator=gen, device="cuda"))
    sigma = ptebd.svd_batched(a)[0]
    norm2 = torch.view_as_real(a).double().square().sum((1, 2, 3))
    change = 0.5 * (sigma.square().sum(1) / norm2 - 1.0)
    assert abs(change.mean().item()) <= 2.0 ** -24 / 16
