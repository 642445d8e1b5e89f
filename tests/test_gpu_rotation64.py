"""The complex128 rotations of the Jacobi SVD are worked out in FP64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ptebd():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_02667_gb300 import ptebd as mod
    return mod


def unitary(rng, n):
    return np.linalg.qr(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))[0]


# One pair of columns: the first sweep makes them orthogonal to the rounding of FP64 (at most
# 0.6 of the threshold 4 sqrt(2) 2^-53 in a numpy model of these matrices), and the second
# finds nothing to rotate.  A tangent of 24 bits leaves 1e5 times the threshold and more.
@pytest.mark.parametrize("seed", range(3))
def test_one_rotation_makes_a_pair_orthogonal(ptebd, seed):
    rng = np.random.default_rng([seed, 0x5EE])
    for _ in range(12):
        a = unitary(rng, 2) @ np.diag([0.8, 0.6]) @ unitary(rng, 2)
        gate = np.concatenate([a.reshape(4, 1), rng.standard_normal((4, 3)) + 0j], axis=1)
        gate = np.linalg.qr(gate)[0]  # a unitary whose first column is the state it makes of |00>
        st = ptebd.State(2, 2, "fp64")
        st.apply_bonds([0], gate[None])
        assert st.svd_sweeps()[0][0] == 2
        assert np.abs(st.lam(0) - [0.8, 0.6]).max() <= 8 * 2.0 ** -53


# Columns whose lengths lie far apart (their squares still normal numbers), and whole matrices
# near the ends of the range.
@pytest.mark.parametrize("low", [0, -20, -100, -140])
@pytest.mark.parametrize("scale", [0, 300, -300])
def test_ranges(ptebd, low, scale):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng([abs(low), abs(scale)])
    rows, cols = 40, 12
    u = np.linalg.qr(rng.standard_normal((rows, cols)) + 1j * rng.standard_normal((rows, cols)))[0]
    # orthogonal columns of length 1 .. 10^low, and a first one that overlaps all others
    length = 10.0 ** np.linspace(0, low, cols)
    a = u * length
    a[:, 0] += 0.3 * u[:, 1:].sum(axis=1)
    a *= 2.0 ** scale
    t = torch.from_numpy(a[None]).cuda()
    sigma, v = ptebd.svd_batched(t, want_u=True)
    sigma, v = sigma[0].cpu().numpy(), v[0].cpu().numpy()
    assert np.all(np.isfinite(sigma)) and np.all(np.diff(sigma) <= 0)
    ref = np.linalg.svd(a, compute_uv=False)
    assert np.abs(sigma - ref).max() <= 1e-13 * ref[0]
    g = np.abs(v.conj().T @ v - np.eye(cols))
    assert g.max() <= 1.5 * 4 * np.sqrt(rows) * 2.0 ** -53
