"""The paths that a size, a batch or a workspace selects, against the oracle and each other:
contractions at the edges of their tiles and at the ends of the chain, truncation below and
above 128 columns with ties, sampling in whole batches, in parts and with the state's scratch,
and an SVD by several thread blocks against the same SVD by one."""
import numpy as np
import pytest

import oracle
from paper_2312_02667_gb300 import inputs

from gpu_helpers import load_into, mini_vidal, to_oracle

pytestmark = pytest.mark.gpu
U64 = 2.0 ** -53


@pytest.fixture(scope="module")
def ptebd():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_02667_gb300 import ptebd as mod
    return mod


def evolved(ptebd, seed, n, chi, prec, depth=9):
    st = ptebd.State(n, chi, prec)
    for parity, _, gates in inputs.brickwork_circuit(seed, n, depth):
        st.apply_layer(gates, parity)
    return st


# Both sides contract the same tensors in FP64, 4 products of chi terms a site: errors add up to
# at most about n * 8 chi roundings of a value of order one, taken with a factor 8.
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n,chi", [(2, 2), (3, 3), (5, 4), (14, 15), (14, 17), (13, 33), (16, 65)])
def test_contractions_at_edges(ptebd, n, chi, prec):
    st, other = evolved(ptebd, 21, n, chi, prec), evolved(ptebd, 22, n, max(2, chi - 1), prec)
    a = to_oracle(st)
    tol = 64 * n * max(chi, 8) * U64
    assert abs(st.norm() - oracle.norm(a)) <= tol
    same = evolved(ptebd, 23, n, chi, prec)
    assert abs(st.overlap(same) - oracle.overlap(a, to_oracle(same))) <= tol
    op = inputs.random_one_site_op(4)
    for j in sorted({0, n // 2, n - 1}):
        assert abs(st.expect(j, op) - oracle.expect_one_site(a, j, op)) <= tol * max(1.0, np.linalg.norm(op, 2))
    op2 = inputs.haar_u4(np.random.default_rng(6))  # (not Hermitian)
    for j in sorted({0, (n - 1) // 2, n - 2}):
        assert abs(st.expect2(j, op2) - oracle.expect_two_site(a, j, op2)) <= tol
    assert abs(other.norm() - oracle.norm(to_oracle(other))) <= tol


# Equal singular values and as many zeros, 2 chi columns: up to 128 are ranked, more are sorted.
@pytest.mark.parametrize("chi", [16, 63, 64, 65, 128])
def test_truncation_with_ties(ptebd, chi):
    rng = np.random.default_rng(chi)
    iso = [np.linalg.qr(rng.standard_normal((2 * chi, chi)) + 1j * rng.standard_normal((2 * chi, chi)))[0]
           for _ in range(2)]
    gb = iso[0].reshape(2, chi, chi)
    gb1 = np.ascontiguousarray(iso[1].conj().T.reshape(chi, 2, chi).transpose(1, 0, 2))
    mps = mini_vidal(np.ones(chi), gb, np.ones(chi), gb1, np.ones(chi))
    ref = oracle.Vidal([g.copy() for g in mps.gammas], [l.copy() for l in mps.lambdas])
    st = ptebd.State(4, chi, "fp64")
    load_into(st, mps)
    gate = np.eye(4, dtype=complex)
    st.apply_bonds([1], gate[None])
    oracle.apply_bonds(ref, [1], gate[None], chi, 1e-12)
    lam, want = st.lam(1), np.asarray(ref.lambdas[1])
    assert len(lam) == len(want) == chi
    # a rotation threshold of 4 sqrt(rows) u leaves sums over chi columns of about this
    assert np.abs(lam - want).max() <= 4 * np.sqrt(2 * chi) * U64 * chi


# The smallest workspace (t and u in the state's scratch), one that holds part of the samples,
# and one that holds all of them: the same bits.
@pytest.mark.parametrize("samples", [1, 40, 130])
def test_sampling_workspaces_agree(ptebd, samples):
    torch = pytest.importorskip("torch")
    n, chi, chip = 12, 15, 16
    st = evolved(ptebd, 31, n, chi, "mixed")
    u = np.random.default_rng(samples).random((samples, n))
    up = lambda x: (x + 255) // 256 * 256
    least = (up(n * chip * chip * 16) + 2 * up(samples * chip * 16) + up(samples * n * 8) + up(samples * n * 4) + 256)
    full = max(least, ptebd.ptebd_sample_workspace_bytes(st.handle, samples))
    want = oracle.sample(to_oracle(st), u)
    for size in {least, (least + full) // 2, full}:
        ws = torch.empty(size, dtype=torch.uint8, device="cuda")
        assert np.array_equal(ptebd.ptebd_sample(st.handle, u, ws), want), size
    with pytest.raises(ptebd.PtebdError):
        ptebd.ptebd_sample(st.handle, u, torch.empty(least - 256, dtype=torch.uint8, device="cuda"))


# Few matrices are each spread over several thread blocks, many are not: the same bits.
@pytest.mark.parametrize("prec,rows,cols", [("mixed", 64, 64), ("mixed", 130, 127), ("mixed", 256, 250),
                                            ("mixed", 300, 50), ("mixed", 400, 60), ("fp64", 64, 61),
                                            ("fp64", 128, 100), ("fp64", 200, 40)])
def test_svd_of_few_and_of_many(ptebd, prec, rows, cols):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(rows + cols)
    z = rng.standard_normal((160, rows, cols)) + 1j * rng.standard_normal((160, rows, cols))
    t = torch.from_numpy(z).to(torch.complex64 if prec == "mixed" else torch.complex128).cuda()
    s, u = ptebd.svd_batched(t, want_u=True)
    for k in (1, 2, 19, 40):
        sk, uk = ptebd.svd_batched(t[:k].contiguous(), want_u=True)
        assert torch.equal(sk, s[:k]) and torch.equal(uk, u[:k]), k
