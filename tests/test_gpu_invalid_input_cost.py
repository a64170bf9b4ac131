"""An invalid factor costs no sweep where a sweep is long (-m gpu): the launches counted are those of
the set-up."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,kw", [(96, {"block_w": 2}), (150, {"block_w": 1, "ordering": "modulus"}),
                                  (80, {"block_w": 4, "precision": "fp32"})])
@pytest.mark.parametrize("cplx", [False, True])
def test_no_sweep_for_an_invalid_factor(cuda_dev, n, kw, cplx):
    import torch

    from paper_1008_0201_gb300 import binding

    G = np.random.default_rng(n).standard_normal((n + 3, n)) + (1j if cplx else 0.0)
    G[n // 2, n // 3] = np.nan
    out = binding.jacobi_eig_pd(torch.from_numpy(G).to(cuda_dev), binding.default_opts(**kw), raise_on_error=False)
    assert out["status"] == binding.JAC_ENONFINITE
    # signs, finiteness, gather, V, pair cache, flags, schedule, FP32 copy
    assert 0 < out["info"]["launches"] <= 8
