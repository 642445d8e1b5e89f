"""complex64 SVDs with and without vectors, which take two kernels.

With vectors: columns are left orthogonal only to 8 sqrt(rows) 2^-24, so the isometry
U S^-1 (U^H A) is 1e-4 off the exact one in a direction that the order of the pairs decides.
The library has always met them in row-cyclic blocks of 16 columns by decreasing norm, and
golden/svd_vectors.npz holds what that order gives.

Without: the layers' kernel, at the edges of its row classes and whatever the batch."""
import os

import numpy as np
import pytest

from test_gpu_jacobi_sizes import SIZES, matrices

pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "svd_vectors.npz")
# one of each height class (up to 32, 64, 128, 256, 512 rows)
VECTORS = [(30, 24), (64, 40), (100, 80), (200, 150), (300, 240)]


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_02667_gb300 import ptebd
    return torch, ptebd


def case(rows, cols):
    """A Ginibre matrix and the two vectors its isometry is applied to."""
    rng = np.random.default_rng([rows, cols, 7])
    a = (rng.standard_normal((rows, cols)) + 1j * rng.standard_normal((rows, cols))) / np.sqrt(2 * rows)
    return a.astype(np.complex64), rng.standard_normal((cols, 2)) / np.sqrt(cols)


def isometry_on(a, probe, sigma, u):
    a, u = a.astype(complex), u.astype(complex)
    return (u / sigma) @ (u.conj().T @ (a @ probe))


# The same pairs in the same order with FP32 rounding: a few 1e-6 at most (another order:
# 1e-4 from 200 rows on).
@pytest.mark.parametrize("rows,cols", VECTORS)
def test_vectors_keep_the_order_of_blocks(env, rows, cols):
    torch, ptebd = env
    a, probe = case(rows, cols)
    sigma, u = ptebd.svd_batched(torch.from_numpy(a[None]).cuda(), want_u=True)
    got = isometry_on(a, probe, sigma[0].cpu().numpy(), u[0].cpu().numpy())
    want = np.load(GOLDEN)[f"{rows}x{cols}"].astype(complex)
    assert np.linalg.norm(got - want) <= 2e-5 * np.linalg.norm(want)


@pytest.mark.parametrize("rows,cols", SIZES)
def test_values_alone_against_lapack(env, rows, cols):
    torch, ptebd = env
    a = matrices(np.random.default_rng([rows, cols, 2]), rows, cols).astype(np.complex64)
    sigma = ptebd.svd_batched(torch.from_numpy(a).cuda(), want_u=False)[0].cpu().numpy()
    for i in range(3):
        ref = np.linalg.svd(a[i].astype(complex), compute_uv=False)
        assert np.abs(sigma[i] - ref).max() <= 1e-5 * ref[0]


# Few matrices are each spread over several thread blocks, many are not: the same bits.
@pytest.mark.parametrize("rows,cols", [(64, 64), (130, 127), (256, 250), (300, 50), (400, 60)])
def test_values_alone_of_few_and_of_many(env, rows, cols):
    torch, ptebd = env
    rng = np.random.default_rng(rows * cols)
    z = rng.standard_normal((160, rows, cols)) + 1j * rng.standard_normal((160, rows, cols))
    t = torch.from_numpy(z).to(torch.complex64).cuda()
    s = ptebd.svd_batched(t, want_u=False)[0]
    for k in (1, 2, 19, 40):
        assert torch.equal(ptebd.svd_batched(t[:k].contiguous(), want_u=False)[0], s[:k]), k
