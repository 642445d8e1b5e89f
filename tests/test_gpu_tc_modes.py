"""ptebd_set_tensor_cores on states whose padded bond dimension (256) reaches the tensor
cores: gated stages (mode 1) and the tSU steps as well (mode 2), against the CUDA cores and
the oracle; and smaller states, which take the CUDA cores in every mode."""
import functools

import numpy as np
import pytest

import oracle
from paper_2312_02667_gb300 import inputs

from gpu_helpers import compare_spectra, fidelity, load_into, to_oracle

pytestmark = pytest.mark.gpu
N, DEPTH = 18, 10


@pytest.fixture(scope="module")
def ptebd():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_02667_gb300 import ptebd as mod
    return mod


@functools.lru_cache(maxsize=None)
def grown(chi):
    """The oracle's state before a layer (its middle bonds at chi), the layer, and the state after it with g = 1."""
    circuit = list(inputs.brickwork_circuit(61, N, DEPTH + 1))
    ref = oracle.product_state(N)
    for parity, _, gates in circuit[:DEPTH]:
        oracle.apply_layer(ref, gates, parity, chi, 1e-12, g=0)
    before = oracle.Vidal([g.copy() for g in ref.gammas], [l.copy() for l in ref.lambdas])
    parity, _, gates = circuit[DEPTH]
    oracle.apply_layer(ref, gates, parity, chi, 1e-12, g=1)
    return before, (parity, gates), ref


def layer(ptebd, before, step, chi, mode):
    st = ptebd.State(N, chi, "mixed", cutoff=1e-12, g=1)
    st.set_tensor_cores(mode)
    load_into(st, before)
    st.apply_layer(step[1], step[0])
    return to_oracle(st)


def same_bits(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a.gammas + a.lambdas, b.gammas + b.lambdas))


# the tolerances of the mixed path against the oracle (one layer and its tSU steps)
@pytest.mark.parametrize("chi", [130, 256])
def test_modes_match_cuda_cores_and_oracle(ptebd, chi):
    before, step, ref = grown(chi)
    assert max(len(l) for l in before.lambdas) > 128
    out = [layer(ptebd, before, step, chi, mode) for mode in (0, 1, 2)]
    assert not same_bits(out[0], out[1]) and not same_bits(out[1], out[2])  # (three sets of kernels)
    for st in out:
        for a, b, c in zip(st.lambdas, ref.lambdas, out[0].lambdas):
            compare_spectra(a, b, 1e-5, 1e-12, chi)
            compare_spectra(a, c, 1e-5, 1e-12, chi)
        assert fidelity(st, ref) >= 1 - 1e-6
        assert fidelity(st, out[0]) >= 1 - 1e-6


@pytest.mark.parametrize("chi", [64, 128])
def test_smaller_states_take_the_cuda_cores(ptebd, chi):
    before, step, _ = grown(chi)
    out = [layer(ptebd, before, step, chi, mode) for mode in (0, 1, 2)]
    assert same_bits(out[0], out[1]) and same_bits(out[0], out[2])
