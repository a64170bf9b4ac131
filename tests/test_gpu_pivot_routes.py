"""The routes of the pivot (-m gpu): one kernel per pivot for few pivots in a step, core and
J-orthogonalization apart for many (the same arithmetic: bit-identical results), and the pivot in
shifted representation for complex problems of order 256 and more."""
import numpy as np
import pytest

from checks import EPS, compare, kappa_A

pytestmark = pytest.mark.gpu

EDGES = {32: (2, 3, 16, 31, 32), 64: (33, 63, 64, 65, 96, 127, 128)}


@pytest.mark.parametrize("km", [32, 64])
@pytest.mark.parametrize("prod", ["split16", "mma"])
def test_many_pivots_equal_few(cuda_dev, km, prod):
    import torch

    from paper_1008_0201_gb300 import binding

    g = np.random.default_rng(77 + km)
    base = []
    for n in EDGES[km]:
        J = np.ones(n, dtype=np.int8)
        J[g.choice(n, size=n // 3, replace=False)] = -1
        base.append((g.standard_normal((n + n // 4, n)), J))
    opts = binding.default_opts(f64_products=prod)

    def solve(problems):
        out, rc = binding.jacobi_eig_batched([torch.from_numpy(G).to(cuda_dev) for G, _ in problems],
                                             [torch.from_numpy(J).to(cuda_dev) for _, J in problems], opts, want_u=True)
        assert rc == 0
        return out

    few = solve(base)
    many = solve(base * (160 // len(base) + 1))  # more than 152 pivots in every step
    for i, out in enumerate(many):
        for key in ("lam", "V", "U"):
            assert torch.equal(out[key], few[i % len(base)][key]), (i, key)
    for (G, J), out in zip(base, few):
        compare(G, J, {k: out[k].cpu().numpy() for k in ("lam", "G", "U", "V")})


@pytest.mark.parametrize("n", [255, 256])
def test_complex_order_at_the_route_limit(cuda_dev, n):
    import torch

    from paper_1008_0201_gb300 import binding

    g = np.random.default_rng(n)
    m = n + 40
    G = g.standard_normal((m, n)) + 1j * g.standard_normal((m, n))
    out = binding.jacobi_eig_pd(torch.from_numpy(G).to(cuda_dev), binding.default_opts())
    ref = np.sort(np.linalg.svd(G, compute_uv=False)) ** 2
    lam, V, Go = (out[k].cpu().numpy() for k in ("lam", "V", "G"))
    assert np.max(np.abs(lam - ref) / ref) <= 50 * n * EPS * kappa_A(G)
    assert np.linalg.norm(V.conj().T @ V - np.eye(n)) <= 100 * n * EPS * 100  # the pairing's 1e-11
    assert np.linalg.norm(G @ V - Go) / np.linalg.norm(G) <= 100 * n * EPS
