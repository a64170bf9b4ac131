"""The backward inside a stream capture (-m gpu)."""
import pytest

pytestmark = pytest.mark.gpu


def test_backward_in_a_capture(cuda_dev):
    import torch

    from paper_1008_0201_gb300 import binding

    g = torch.Generator(device=cuda_dev)
    g.manual_seed(3)
    rand = lambda *s: torch.randn(*s, generator=g, device=cuda_dev, dtype=torch.float64)  # noqa: E731
    n, batch = 40, 3
    lam = torch.cumsum(0.2 + rand(batch, n).abs(), 1)
    U = torch.linalg.qr(rand(batch, n, n))[0]
    lam_bar, U_bar = rand(batch, n), rand(batch, n, n)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        H = binding.jacobi_eig_backward(lam, U, lam_bar, U_bar)[0]
    for _ in range(2):  # the captured call reads its inputs again at every replay
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(H, binding.jacobi_eig_backward(lam, U, lam_bar, U_bar)[0])
        U_bar.mul_(-0.5)

