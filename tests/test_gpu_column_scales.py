"""Column norms far apart and far from 1 (-m gpu): ratios up to 1e24 inside one pivot block against the
oracle, and factors whose squared norms leave FP32's normal range."""
import numpy as np
import pytest

from checks import EPS32, compare, to_np

pytestmark = pytest.mark.gpu


def factor(n, ratio, signs):
    g = np.random.default_rng(n)
    D = np.where(g.permutation(n) < n // 2, ratio ** -0.5, ratio ** 0.5)
    J = np.ones(n, dtype=np.int8)
    if signs == "opposite":
        J[g.choice(n, size=n // 3, replace=False)] = -1
    return g.standard_normal((n + 8, n)) * D, J


@pytest.mark.parametrize("ratio", [1e12, 1e17, 2e18, 1e20, 1e24])
@pytest.mark.parametrize("signs", ["same", "opposite"])
@pytest.mark.parametrize("n", [24, 64])
def test_norms_far_apart(cuda_dev, n, ratio, signs):
    import torch

    import oracle
    from paper_1008_0201_gb300 import binding

    G, J = factor(n, ratio, signs)
    ref = oracle.solve(G, J)
    for mode in ("full", "oriented"):
        for prec in ("fp64", "fp32", "fp32_only"):
            out = binding.jacobi_hsvd(torch.from_numpy(G).to(cuda_dev), torch.from_numpy(J).to(cuda_dev),
                                      binding.default_opts(block_mode=mode, precision=prec))
            assert out["info"]["sweeps"] <= 16, (mode, prec)
            kw = dict(eps=EPS32) if prec == "fp32_only" else {}
            compare(G, J, to_np(out), ref=ref, check_vectors=prec != "fp32_only", **kw)


@pytest.mark.parametrize("scale", [1e-20, 1e-19, 1e-12, 1e12])
@pytest.mark.parametrize("signs", ["same", "opposite"])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_norms_far_from_one(cuda_dev, scale, signs, prec):
    import torch

    import oracle
    from paper_1008_0201_gb300 import binding

    n = 24
    G, J = factor(n, 1.0, signs)
    ref = oracle.solve(G, J)
    out = binding.jacobi_hsvd(torch.from_numpy(G * scale).to(cuda_dev), torch.from_numpy(J).to(cuda_dev),
                              binding.default_opts(precision=prec))
    lam = out["lam"].cpu().numpy() / scale / scale
    # an FP32 product is resolved to 2^-149: scaled entries below 2^-149 / a_ii are not seen, and n of them
    # move an eigenvalue by n times that (relative) at most; above FP32's subnormals the usual bound
    unseen = 2.0 ** -149 / (scale * scale * np.min(np.sum(G * G, axis=0)))
    kappa = np.linalg.cond(G / np.linalg.norm(G, axis=0)) ** 2
    assert np.max(np.abs(lam - ref["lam"]) / np.abs(ref["lam"])) <= 50 * n * 2.0 ** -53 * kappa + n * kappa * unseen
