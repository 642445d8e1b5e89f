"""States are made and destroyed while a stream of the same thread captures a graph."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_02667_gb300 import ptebd
    return torch, ptebd


def test_states_come_and_go_during_a_capture(env):
    torch, ptebd = env
    old = ptebd.State(8, 8, "mixed")
    old.sync()
    cfg = ptebd.make_config(6, 4, "mixed", 1e-12, 0, "schmidt", -1.0)
    sb, wb, _ = ptebd.ptebd_required_bytes(cfg)
    state, ws = (torch.empty(b, dtype=torch.uint8, device="cuda") for b in (sb, wb))
    side = torch.cuda.Stream()
    x = torch.arange(1000.0, device="cuda")
    y = torch.zeros_like(x)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        torch.mul(x, 2.0, out=y)
        new = ptebd.ptebd_create(cfg, state.data_ptr(), sb, ws.data_ptr(), wb, side.cuda_stream)
        old.close()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, 2.0 * x)
    assert list(ptebd.ptebd_get_chi(new, 6)) == [1] * 5
    ptebd.ptebd_destroy(new)
