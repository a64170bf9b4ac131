"""Invalid factors and signs (-m gpu): refused with the same codes on every route (no sweep, sweeps
launched directly, sweeps as a graph, a schedule by weights, complex), nothing written for invalid
signs, and the next solve is right; and the scratch the library keeps is given back and taken again."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _raw(binding, torch, dev, G, J, **kw):
    n = G.shape[1]
    cplx = np.iscomplexobj(G)
    Gd = torch.from_numpy(np.ascontiguousarray(G.T)).to(dev)
    Jd = torch.from_numpy(J).to(dev)
    lam = torch.full((n,), 7.0, dtype=torch.float64, device=dev)
    U, V = torch.full_like(Gd, 7.0), torch.full((n, n), 7.0, dtype=Gd.dtype, device=dev)
    opts = binding.default_opts(**kw)
    rc, _ = binding.jacobi_hsvd_raw(G.shape[0], n, Gd.data_ptr(), G.shape[0], Jd.data_ptr(), opts, lam.data_ptr(),
                                    U.data_ptr(), G.shape[0], V.data_ptr(), n,
                                    torch.cuda.current_stream().cuda_stream,
                                    binding.JAC_C128 if cplx else binding.JAC_R64)
    torch.cuda.synchronize()
    return rc, Gd.cpu().numpy().T, [t.cpu().numpy() for t in (lam, U, V)]


@pytest.mark.parametrize("n,kw", [(1, {}), (24, {}), (24, {"block_w": 4}), (150, {}),
                                  (150, {"ordering": "cycle_weight"}),
                                  (150, {"precision": "fp32_only"}), (150, {"precision": "fp32"})])
@pytest.mark.parametrize("cplx", [False, True])
def test_invalid_input_is_refused(cuda_dev, n, kw, cplx):
    import torch

    from paper_1008_0201_gb300 import binding

    g = np.random.default_rng(n)
    G = g.standard_normal((n + 3, n)) + (1j * g.standard_normal((n + 3, n)) if cplx else 0.0)
    J = np.ones(n, dtype=np.int8)
    J[n // 2:] = -1
    if cplx and "precision" in kw:
        pytest.skip("complex problems are FP64")
    good = _raw(binding, torch, cuda_dev, G, J, **kw)
    assert good[0] == 0
    for bad in (0, 3, -2):
        Jb = J.copy()
        Jb[n - 1] = bad
        rc, Gout, outs = _raw(binding, torch, cuda_dev, G, Jb, **kw)
        assert rc == -6
        assert np.array_equal(Gout, G) and all((o == 7.0).all() for o in outs)
    for bad in (np.nan, np.inf, -np.inf):
        Gb = G.copy()
        Gb[n // 3, n - 1] = bad
        assert _raw(binding, torch, cuda_dev, Gb, J, **kw)[0] == binding.JAC_ENONFINITE
    again = _raw(binding, torch, cuda_dev, G, J, **kw)
    assert again[0] == 0 and np.array_equal(again[1], good[1])
    assert all(np.array_equal(a, b) for a, b in zip(again[2], good[2]))


def test_scratch_is_given_back(cuda_dev):
    import torch

    from paper_1008_0201_gb300 import binding

    lib = binding.load_library()
    G = np.random.default_rng(3).standard_normal((80, 64))
    J = np.ones(64, dtype=np.int8)
    first = _raw(binding, torch, cuda_dev, G, J)
    for _ in range(2):
        assert lib.jacobi_release_scratch() == 0
        out = _raw(binding, torch, cuda_dev, G, J)
        assert out[0] == 0 and np.array_equal(out[2][0], first[2][0])
