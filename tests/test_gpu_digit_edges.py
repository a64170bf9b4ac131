"""The digit Gram and update at the edges of their tiles (-m gpu, against the oracle): pivot blocks of
every remainder of 8 and 16 columns, rows around the 64- and 128-row groups, one CTA or a cluster."""
import numpy as np
import pytest

from checks import compare, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 7, 8, 9, 15, 16, 17, 31, 33, 47, 48, 49, 63, 64])
@pytest.mark.parametrize("m", [64, 65, 127, 129, 300])
def test_one_block(cuda_dev, m, n):
    import torch

    from paper_1008_0201_gb300 import binding

    g = np.random.default_rng(1000 * m + n)
    G = g.standard_normal((m, n))
    J = np.ones(n, dtype=np.int8)
    J[: n // 3] = -1
    out = binding.jacobi_hsvd(torch.from_numpy(G).to(cuda_dev), torch.from_numpy(J).to(cuda_dev))
    assert out["status"] == 0
    compare(G, J, to_np(out))
