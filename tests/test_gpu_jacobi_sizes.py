"""The Jacobi SVD kernel at the sizes where its choices change: rows per lane
(32, 64, 96, 128, 192, 256, 384, 512 rows), matrices that stay in shared memory and matrices
streamed through it, column counts that leave a partial last group, fewer
groups than warps, and rank-deficient and graded columns, through svd_batched
against LAPACK in complex128."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# (rows, cols): the edges of each row class, one past them, and thin matrices of each
SIZES = [(2, 1), (6, 5), (32, 32), (34, 33), (64, 64), (64, 3), (66, 65), (96, 95), (98, 98), (102, 102), (128, 128), (128, 9),
         (130, 127), (192, 190), (194, 60), (200, 130), (256, 103), (256, 105), (256, 256), (258, 50), (258, 255), (300, 111), (384, 100), (386, 90), (512, 17),
         (512, 210)]
U = {"mixed": 2.0 ** -24, "fp64": 2.0 ** -53}
K = {"mixed": 8.0, "fp64": 4.0}  # the rotation threshold: |a^H b| <= K sqrt(rows) u |a| |b|


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_02667_gb300 import ptebd
    return torch, ptebd


def matrices(rng, rows, cols):
    z = rng.standard_normal((3, rows, cols)) + 1j * rng.standard_normal((3, rows, cols))
    z /= np.sqrt(2 * rows)
    z[1] *= 10.0 ** (-3.0 * np.arange(cols) / cols)          # columns of very different length
    if cols >= 3:
        z[2, :, -1] = z[2, :, 0] - 0.5 * z[2, :, 1]          # dependent columns
        z[2, :, cols // 2] = 0.0                             # and a zero one
    return z


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("rows,cols", SIZES)
def test_sizes_against_lapack(env, prec, rows, cols):
    torch, ptebd = env
    a = matrices(np.random.default_rng([rows, cols]), rows, cols)
    t = torch.from_numpy(a).to(torch.complex64 if prec == "mixed" else torch.complex128).cuda()
    sig, u = ptebd.svd_batched(t, want_u=True)
    sig, u = sig.cpu().numpy(), u.cpu().numpy().astype(complex)
    seen = t.cpu().numpy().astype(complex)
    tol = {"mixed": 1e-5, "fp64": 1e-12}[prec]
    orth = 1.5 * K[prec] * np.sqrt(rows) * U[prec]
    for i in range(3):
        ref = np.linalg.svd(seen[i], compute_uv=False)
        assert np.abs(sig[i] - ref).max() <= tol * ref[0]
        # the vectors of values above the rounding of the columns (a value at u sigma_1 has none of its own)
        k = int(np.sum(ref > 1e3 * U[prec] * ref[0]))
        g = np.abs(u[i][:, :k].conj().T @ u[i][:, :k] - np.eye(k))
        assert g.max() <= orth, (i, g.max() / orth)


def test_repeats_bitwise_and_batch_order(env):
    # the warps of a matrix hand groups on in a fixed order, whatever their timing
    torch, ptebd = env
    rng = np.random.default_rng(5)
    a = rng.standard_normal((160, 96, 90)) + 1j * rng.standard_normal((160, 96, 90))
    t = torch.from_numpy(a).to(torch.complex64).cuda()
    s0, u0 = ptebd.svd_batched(t, want_u=True)
    s1, u1 = ptebd.svd_batched(t.flip(0).contiguous(), want_u=True)
    assert torch.equal(s0, s1.flip(0)) and torch.equal(u0, u1.flip(0))
