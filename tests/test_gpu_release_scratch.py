"""The scratch kept between calls goes back to the device (-m gpu)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_release(cuda_dev):
    import torch

    from paper_1008_0201_gb300 import binding

    G = torch.from_numpy(np.random.default_rng(5).standard_normal((640, 512))).to(cuda_dev)
    first = binding.jacobi_eig_pd(G)["lam"]
    torch.cuda.synchronize()
    kept = torch.cuda.mem_get_info(cuda_dev)[0]
    binding.jacobi_release_scratch()
    assert torch.cuda.mem_get_info(cuda_dev)[0] > kept  # 2 x 2.6 MB of G and V alone
    assert torch.equal(binding.jacobi_eig_pd(G)["lam"], first)
