"""The two digit Gram kernels (-m gpu): the tensor-memory one and the mma.sync one give the same bits
at the edges of their tiles, stages and row counts, and the former is right where one CTA takes two
shares of the rows."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# (m, n): one pivot block of 33..64 columns (32 and less: the other capacity); rows below, at and
# above one and two stages of 128
SHAPES = [(33, 33), (48, 47), (64, 64), (112, 49), (113, 64), (128, 64), (129, 63), (144, 64), (145, 50), (256, 64),
          (257, 64), (400, 33), (40, 24), (128, 32), (130, 32), (300, 17)]


def test_same_bits(cuda_dev):
    import torch

    from paper_1008_0201_gb300 import binding

    g = np.random.default_rng(11)
    Gs = [g.standard_normal(s) * 10.0 ** g.uniform(-3, 3, size=s[1]) for s in SHAPES]
    Js = [np.where(np.arange(s[1]) % 3 == 2, -1, 1).astype(np.int8) for s in SHAPES]
    outs = []
    for prod in ("split16", "split16_tc"):
        for G, J in zip(Gs, Js):  # one problem per call: the rows of the class are its own
            out, rc = binding.jacobi_eig_batched([torch.from_numpy(G).to(cuda_dev)], [torch.from_numpy(J).to(cuda_dev)],
                                                 binding.default_opts(f64_products=prod), want_u=True)
            assert rc == 0
            outs.append(out[0])
    for s, x, y in zip(SHAPES, outs, outs[len(SHAPES):]):
        for key in ("lam", "U", "V"):
            assert torch.equal(x[key], y[key]), (s, key)


def test_two_shares_per_block(cuda_dev):
    import torch

    from paper_1008_0201_gb300 import binding

    m, n = 1500, 1300  # 21 pairs, 8 shares each: more than 152
    G = np.random.default_rng(12).standard_normal((m, n))
    out = binding.jacobi_eig_pd(torch.from_numpy(G).to(cuda_dev))
    want = np.sort(np.linalg.svd(G, compute_uv=False) ** 2)
    got = out["lam"].cpu().numpy()
    # rounding of a Gram entry or a rotation: n eps ||G||^2 at most, over ~10 sweeps, factor 6
    assert np.abs(got - want).max() <= 60 * n * 1.1e-16 * want[-1]
