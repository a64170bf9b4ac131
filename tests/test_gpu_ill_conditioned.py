"""Pivot blocks beyond what FP32 factors (-m gpu, against the oracle): the two-float Cholesky takes
them (scaled Schur pivots down to 2^-36), the FP64 pivot below that."""
import numpy as np
import pytest

from checks import compare, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("angle", [2e-3, 1e-4, 1e-5, 2e-6])  # Schur pivots 4e-6 .. 4e-12
@pytest.mark.parametrize("n,w", [(20, 10), (31, 16), (47, 32), (64, 32)])
@pytest.mark.parametrize("factor,signs", [("chol", "same"), ("chol_diagpiv", "opposite"), ("chol_signpiv", "same"),
                                          ("chol_signpiv", "opposite")])
def test_nearly_parallel_columns(cuda_dev, n, w, angle, factor, signs):
    import torch

    from paper_1008_0201_gb300 import binding

    g = np.random.default_rng(n)
    G = g.standard_normal((n + 9, n)) * 10.0 ** g.uniform(-3, 3, n)  # columns of very different size
    i, j = 2, n - 3
    G[:, j] = G[:, i] + angle * np.linalg.norm(G[:, i]) / np.sqrt(n + 9) * g.standard_normal(n + 9)
    J = np.ones(n, dtype=np.int8)
    J[g.choice(n, size=n // 3, replace=False)] = -1
    J[i] = 1
    J[j] = 1 if signs == "same" else -1
    out = binding.jacobi_hsvd(torch.from_numpy(G).to(cuda_dev), torch.from_numpy(J).to(cuda_dev),
                              binding.default_opts(block_w=w, factor=factor))
    assert out["status"] == 0
    # without the vectors: the vector bound of checks.py divides by the relative gap, which is up to 1e10
    # for the small eigenvalue of the pair, below what any FP64 solver (the oracle included) resolves
    compare(G, J, to_np(out), check_vectors=False)
