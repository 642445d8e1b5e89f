"""Several threads that read one state at a time: each gets what it asked for."""
import threading

import numpy as np
import pytest

from paper_2312_02667_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ptebd():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_02667_gb300 import ptebd as mod
    return mod


def test_threads_read_one_state(ptebd):
    n = 24
    st = ptebd.State(n, 16, "mixed")
    for parity, _, gates in inputs.brickwork_circuit(71, n, 8):
        st.apply_layer(gates, parity)
    lam = [st.lam(b) for b in range(n - 1)]
    assert len({v.tobytes() for v in lam}) == n - 1  # (no two bonds alike)
    stats = st.bond_stats()
    wrong = []

    def read(k):
        rng = np.random.default_rng(k)
        for _ in range(200):
            b = int(rng.integers(n - 1))
            if not np.array_equal(st.lam(b), lam[b]):
                wrong.append(("lam", b))
            if k % 4 == 0 and not all(np.array_equal(x, y) for x, y in zip(st.bond_stats(), stats)):
                wrong.append("stats")

    threads = [threading.Thread(target=read, args=(k,)) for k in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
