"""The choice of the digit Gram (-m gpu): factors on both sides of each of its lines (rows per share, one or
two shares per CTA, more clusters than run at once, narrow pairs, batches) against LAPACK."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(3072, 64), (3088, 64), (2304, 576), (2048, 640), (2064, 640), (2304, 1024), (3400, 231)])
def test_single(cuda_dev, m, n):
    import torch

    from paper_1008_0201_gb300 import binding

    G = np.random.default_rng(m + n).standard_normal((m, n))
    out = binding.jacobi_eig_pd(torch.from_numpy(G).to(cuda_dev), binding.default_opts(want_v=0))
    want = np.sort(np.linalg.svd(G, compute_uv=False) ** 2)
    # rounding of a Gram entry or a rotation: n eps ||G||^2 at most, over ~10 sweeps, factor 6
    assert np.abs(out["lam"].cpu().numpy() - want).max() <= 60 * n * 1.1e-16 * want[-1]


@pytest.mark.parametrize("m,n", [(192, 64), (193, 64), (260, 60), (260, 61), (260, 122)])
def test_batch(cuda_dev, m, n):
    import torch

    from paper_1008_0201_gb300 import binding

    G = np.random.default_rng(m + n).standard_normal((160, m, n))
    out = binding.jacobi_eig_batched_uniform(torch.from_numpy(G).to(cuda_dev), opts=binding.default_opts(want_v=0))
    want = np.sort(np.linalg.svd(G, compute_uv=False) ** 2, axis=1)
    assert np.abs(out["lam"].cpu().numpy() - want).max() <= 60 * n * 1.1e-16 * want.max()
