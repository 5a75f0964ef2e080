"""The training kernel of one block, which runs where the cluster of eight does
not fit: the cluster's results bit for bit, from any number of earlier steps."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from gpu_util import DEV  # noqa: E402
from paper_2007_01277_gb300 import costmodel as CM  # noqa: E402
from paper_2007_01277_gb300 import hfuse as H  # noqa: E402


@pytest.mark.parametrize("batch", [1, 3, 32, 33, 64])
def test_same_bits_as_the_cluster(batch):
    g = torch.Generator().manual_seed(batch)
    X, Y = torch.rand(200, 24, generator=g).to(DEV), torch.rand(200, generator=g).to(DEV)
    idx = torch.randint(0, 200, (5 * batch,), generator=g, dtype=torch.int32).to(DEV)
    out = []
    for train in (H.hf_mlp_train, H.hf_mlp_train_block):
        P = CM.xavier_params(batch).to(DEV)
        M, V = torch.full_like(P, 1e-3), torch.full_like(P, 1e-5)
        loss, grad = torch.empty(5, device=DEV), torch.empty_like(P)
        train(P, M, V, X, Y, idx, 5, batch, t0=7, loss_out=loss, grad_out=grad)
        torch.cuda.synchronize()
        out.append((P, M, V, loss, grad))
    for a, b in zip(*out):
        assert torch.equal(a, b)
    for bad in (dict(steps=-1), dict(batch=65), dict(batch=0)):
        with pytest.raises(H.HFError):
            H.hf_mlp_train_block(P, M, V, X, Y, idx, **{"steps": 1, "batch": batch, **bad})


def test_captured_run_keeps_the_cluster():
    """Recorded into a graph the run is the cluster's too: one block would take
    more than four times as long."""
    g = torch.Generator().manual_seed(1)
    X, Y = torch.rand(200, 24, generator=g).to(DEV), torch.rand(200, generator=g).to(DEV)
    idx = torch.randint(0, 200, (6400,), generator=g, dtype=torch.int32).to(DEV)
    P = CM.xavier_params(1).to(DEV)
    M, V = torch.zeros_like(P), torch.zeros_like(P)
    direct = [t.clone() for t in (P, M, V)]
    H.hf_mlp_train(*direct, X, Y, idx, 100, 64)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        H.hf_mlp_train(P, M, V, X, Y, idx, 100, 64)
    graph.replay()
    torch.cuda.synchronize()
    for a, b in zip((P, M, V), direct):
        assert torch.equal(a, b)

    def best(fn):
        times = []
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            fn()
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)

    assert best(graph.replay) < 2 * best(lambda: H.hf_mlp_train(P, M, V, X, Y, idx, 100, 64))
    assert 2 * best(graph.replay) < best(lambda: H.hf_mlp_train_block(P, M, V, X, Y, idx, 100, 64))
