"""The workloads whose speed is measured: what programs have this library do, through its public
entry points (paper_1008_0201_gb300.binding and .autograd), over the sizes its benchmark
configurations and tests use.

A case names its entry point in "kind":
  single   jacobi_hsvd / jacobi_eig_pd on one factor G (real or complex), eigenvalues, U and
           (unless v = 0) V returned;
  batched  jacobi_eig_batched_raw on `count` problems of uneven order in flat buffers;
  train    one training step through autograd.eigh_factor: forward, loss, gradient of G;
  backward jacobi_eig_backward alone (H_bar of a stack of eigendecompositions).

Eigenvectors are defined up to a sign (a phase when complex).  As a program that stores or
compares them does, run() fixes it: the first component of every column of U is made real and
nonnegative and the column of V goes with it.
"""
import math

import numpy as np
import torch

from paper_1008_0201_gb300 import autograd, binding


def listed():
    single = dict(kind="single", cplx=0, grade=0, v=1)
    return [
        # one tiny problem: a caller that solves small matrices one at a time; launches and host work
        dict(single, name="pd_24_one_block", m=24, n=24, neg=0.0, w=32, order="round_robin", mode="full",
             factor="chol_signpiv", prec="fp64"),
        # the plain positive definite configuration: cyclic (modulus) ordering, width 8
        dict(single, name="pd_64_modulus", m=64, n=64, neg=0.0, w=8, order="modulus", mode="full",
             factor="chol_signpiv", prec="fp64"),
        # the hyperbolic configuration in its fastest form: block-oriented, FP32 sweeps + FP64 polish
        dict(single, name="hsvd_512_mixed", m=512, n=512, neg=0.5, w=32, order="round_robin", mode="oriented",
             factor="chol_signpiv", prec="fp32"),
        # the same problem with the paper's per-cycle largest-weight pivoting, FP64 throughout
        dict(single, name="hsvd_512_weight", m=512, n=512, neg=0.5, w=32, order="cycle_weight", mode="full",
             factor="chol_signpiv", prec="fp64"),
        # a tall data factor of ragged sizes, default options, left vectors only
        dict(single, name="tall_1237x301", m=1237, n=301, neg=0.4, w=32, order="round_robin", mode="full",
             factor="chol_signpiv", prec="fp64", v=0),
        # a large indefinite problem of odd order (the paper's order range on one GPU), mixed precision
        dict(single, name="hsvd_1501_mixed", m=1501, n=1501, neg=0.5, w=32, order="round_robin",
             mode="oriented", factor="chol_signpiv", prec="fp32"),
        # the graded complex Hermitian configuration at a quarter of its order, mixed precision (a few
        # more rows than columns, so that the vectors of the small end are determined to 1e-10)
        dict(single, name="graded_complex_1024", m=1152, n=1024, neg=0.0, w=32, order="round_robin",
             mode="oriented", factor="chol_signpiv", prec="fp32", cplx=1, grade=8),
        # a complex hyperbolic problem, default options in FP64
        dict(single, name="complex_201_fp64", m=233, n=201, neg=0.4, w=32, order="round_robin", mode="full",
             factor="chol_signpiv", prec="fp64", cplx=1),
        # the batched configuration: thousands of indefinite problems of orders 8..128, with V
        dict(kind="batched", name="batched_4000_fp64", count=4000, lo=8, hi=128, tall=1.0, neg=0.3, prec="fp64"),
        # squared singular values of many small well-conditioned factors in FP32 (screening)
        dict(kind="batched", name="batched_4000_fp32", count=4000, lo=8, hi=128, tall=1.5, neg=0.0,
             prec="fp32_only"),
        # a training step of the differentiation configuration
        dict(kind="train", name="train_96x256", count=96, n=256, neg=0.0),
        # its backward alone, at full batch: H_bar from stored eigenpairs
        dict(kind="backward", name="backward_256x256", count=256, n=256),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["single", "single", "single", "complex", "batched", "batched", "train", "backward"])
    mode = rng.choice(["full", "oriented"])
    order = rng.choice(["round_robin", "round_robin", "modulus_mod", "cycle_weight"] + ["modulus"] * (mode == "full"))
    factor = rng.choice(["chol", "chol_diagpiv", "chol_signpiv", "chol_signpiv"])
    prec = rng.choice(["fp64", "fp32"])
    if kind == "single":
        n = _log(rng, 12, 900)
        m = n + rng.randrange(0, n + 1) if rng.random() < 0.5 else n
        return dict(kind="single", cplx=0, grade=0, v=rng.choice([1, 1, 0]), m=m, n=n,
                    neg=rng.choice([0.0, 0.3, 0.5]), w=rng.choice([8, 16, 27, 32, 32]) if n < 300 else 32,
                    order=order, mode=mode, factor=factor, prec=prec)
    if kind == "complex":
        n = _log(rng, 16, 400)
        grade = rng.choice([0, 0, 8])
        return dict(kind="single", cplx=1, grade=grade, v=1, m=n + n // 8 + rng.randrange(0, n // 2 + 1), n=n,
                    neg=0.0 if grade else rng.choice([0.0, 0.4]), w=32, order="round_robin", mode=mode,
                    factor="chol_signpiv", prec=prec)
    if kind == "batched":
        lo = _log(rng, 4, 64)
        p = rng.choice(["fp64", "fp32_only"])
        return dict(kind="batched", count=_log(rng, 50, 3000), lo=lo, hi=rng.randrange(lo + 1, 129),
                    tall=1.5 if p == "fp32_only" else rng.choice([1.0, 1.25]),
                    neg=0.0 if p == "fp32_only" else rng.choice([0.0, 0.3]), prec=p)
    n = _log(rng, 32, 256)
    return dict(kind=kind, count=_log(rng, 4, 96), n=n, **({"neg": 0.0} if kind == "train" else {}))


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _signs(n, neg, seed):
    """n signs, round(neg n) of them -1 at random positions."""
    J = np.ones(n, dtype=np.int8)
    k = int(round(neg * n))
    if k:
        J[np.random.default_rng(seed).choice(n, size=k, replace=False)] = -1
    return J


def _orders(case, seed):
    """Orders spread evenly over lo..hi, in an order that depends on the seed, and row counts."""
    span = case["hi"] - case["lo"] + 1
    n = case["lo"] + (np.arange(case["count"], dtype=np.int64) * span) // case["count"]
    if seed is not None:
        n = np.random.default_rng(seed).permutation(n)
    return n, np.ceil(case["tall"] * n).astype(np.int64)


def _opts(case):
    return binding.default_opts(block_w=case["w"], ordering=case["order"], block_mode=case["mode"],
                                factor=case["factor"], precision=case["prec"], want_v=case["v"])


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "single":
        m, n = case["m"], case["n"]
        G = _randn(g, m, n)
        if case["cplx"]:
            G = torch.complex(G, _randn(g, m, n)) * math.sqrt(0.5)
        if case["grade"]:  # column norms fall by 10^-grade over the columns
            G = G * torch.pow(10.0, -case["grade"] * torch.arange(n, device="cuda", dtype=torch.float64) / n)
        J = torch.from_numpy(_signs(n, case["neg"], seed)).cuda()
        return dict(kind=kind, G=G, J=J if case["neg"] else None, opts=_opts(case))
    if kind == "batched":
        n, m = _orders(case, seed)
        goff, voff, loff = (np.concatenate([[0], np.cumsum(x)]) for x in (m * n, n * n, n))
        J = np.concatenate([_signs(int(k), case["neg"], seed + 31 * i) for i, k in enumerate(n)])
        st = dict(kind=kind, n=n.astype(np.int32), m=m.astype(np.int32), G0=_randn(g, int(goff[-1])),
                  J=torch.from_numpy(J).cuda(), goff=goff[:-1].astype(np.uint64),
                  voff=voff[:-1].astype(np.uint64), loff=loff[:-1].astype(np.uint64), v=case["prec"] == "fp64",
                  opts=binding.default_opts(precision=case["prec"], want_v=int(case["prec"] == "fp64")))
        st["G"] = torch.empty_like(st["G0"])
        st["lam"] = torch.empty(int(loff[-1]), device="cuda", dtype=torch.float64)
        if st["v"]:  # where each column of V starts, and the column of every entry
            st["V"] = torch.empty(int(voff[-1]), device="cuda", dtype=torch.float64)
            rep = torch.from_numpy(np.repeat(n, n)).cuda()
            st["head"] = torch.cumsum(rep, 0) - rep
            st["col"] = torch.repeat_interleave(torch.arange(int(loff[-1]), device="cuda"), rep)
        return st
    count, n = case["count"], case["n"]
    if kind == "train":
        return dict(kind=kind, G=_randn(g, count, n, n) / math.sqrt(n), w=_randn(g, n),
                    C=_randn(g, n, 4), opts=binding.default_opts(want_v=0))
    U = torch.linalg.qr(_randn(g, count, n, n))[0]
    lam = torch.cumsum(0.2 + torch.rand(count, n, generator=g, device="cuda", dtype=torch.float64), 1)
    return dict(kind=kind, lam=lam, U=U, lam_bar=_randn(g, count, n), U_bar=_randn(g, count, n, n))


def _phase(U):
    """What makes the first component of every column real and nonnegative."""
    u = U[..., :1, :]
    if U.is_complex():
        return torch.conj(torch.sgn(u))
    return torch.where(u < 0, -1.0, 1.0).to(U.dtype)


def run(s):
    kind = s["kind"]
    if kind == "single":
        out = binding.jacobi_eig_pd(s["G"], s["opts"]) if s["J"] is None else binding.jacobi_hsvd(s["G"], s["J"], s["opts"])
        f = _phase(out["U"])
        r = dict(lam=out["lam"], U=out["U"] * f)
        if out["V"] is not None:
            r["V"] = out["V"] * f
        return r
    if kind == "batched":
        s["G"].copy_(s["G0"])  # the solver works in place
        at = lambda t, off, size: np.uint64(t.data_ptr()) + off * np.uint64(size)  # noqa: E731
        rc, _ = binding.jacobi_eig_batched_raw(
            s["m"], s["n"], at(s["G"], s["goff"], 8), s["m"], at(s["J"], s["loff"], 1), s["opts"],
            at(s["lam"], s["loff"], 8), None, None, at(s["V"], s["voff"], 8) if s["v"] else None,
            s["n"] if s["v"] else None, torch.cuda.current_stream().cuda_stream, want_info=False)
        if rc != binding.JAC_OK:
            raise binding.JacobiError(rc, binding.status_string(rc))
        if not s["v"]:
            return dict(lam=s["lam"].float())  # FP32 results
        V = s["V"]
        f = torch.where(V[s["head"]] < 0, -1.0, 1.0).to(V.dtype)
        return dict(lam=s["lam"], V=V * f[s["col"]])
    if kind == "train":
        G = s["G"].detach().requires_grad_(True)
        lam, U = autograd.eigh_factor(G, None, s["opts"])
        loss = (lam * s["w"]).sum() + (U[:, :, -8:].transpose(-1, -2) @ s["C"]).square().sum()
        loss.backward()
        U = U.detach()
        return dict(lam=lam.detach(), U=U * _phase(U), grad=G.grad)
    return dict(H_bar=binding.jacobi_eig_backward(s["lam"], s["U"], s["lam_bar"], s["U_bar"])[0])


def work(case):
    # Bytes: the factor in, eigenvalues, vectors (and the overwritten factor) out.  Operations: six
    # sweeps of pointwise one-sided Jacobi (n^2/2 pairs: a dot product and two rotated columns).
    if case["kind"] == "single":
        m, n = case["m"], case["n"]
        c = 2 if case["cplx"] else 1
        return {"bytes": 8.0 * c * (3 * m * n + case["v"] * n * n) + 8.0 * n,
                "flops": 6.0 * c * c * n * n * (4 * m + 3 * n * case["v"])}
    if case["kind"] == "batched":
        n, m = (x.astype(np.float64) for x in _orders(case, None))
        v = 1.0 if case["prec"] == "fp64" else 0.0
        return {"bytes": float(np.sum(8.0 * (2 * m * n + v * n * n + n))),
                "flops": float(np.sum(6.0 * n * n * (4 * m + 3 * n * v)))}
    b, n = float(case["count"]), float(case["n"])
    if case["kind"] == "train":  # forward without V, then U^T U_bar, U K, (U K) U^T, H_bar G
        return {"bytes": 8.0 * b * (5 * n * n + 3 * n), "flops": b * (24.0 * n ** 3 + 7.0 * n ** 3)}
    return {"bytes": 8.0 * b * (3 * n * n + 2 * n), "flops": 5.0 * b * n ** 3}


def _adjoint(lam, U, lam_bar, U_bar):
    F = lam.unsqueeze(-2) - lam.unsqueeze(-1)
    F = torch.where(F == 0, torch.zeros_like(F), 1.0 / F)
    K = torch.diag_embed(lam_bar) + F * (U.transpose(-1, -2) @ U_bar)
    return U @ ((K + K.transpose(-1, -2)) / 2) @ U.transpose(-1, -2)


def exact(case, seed):
    s = prepare(case, seed)
    if case["kind"] == "single":
        G = s["G"]
        J = torch.ones(case["n"], device="cuda", dtype=torch.float64) if s["J"] is None else s["J"].double()
        lam, Q = torch.linalg.eigh((G * J) @ G.mH)
        if case["m"] > case["n"]:  # the eigenvalues that are not the m - n zeros
            keep = torch.sort(torch.argsort(lam.abs(), descending=True)[: case["n"]])[0]
            lam, Q = lam[keep], Q[:, keep]
        if case["grade"]:  # a dense eigensolver has the small end of a graded spectrum to norm accuracy only
            return dict(lam=lam, U=None, V=None)
        U = Q * _phase(Q)
        r = dict(lam=lam, U=U)
        if case["v"]:  # G V = U |lam|^(1/2)
            r["V"] = torch.linalg.lstsq(G, U * lam.abs().sqrt()).solution
        return r
    if case["kind"] == "batched":
        n, m, G, J = s["n"].astype(int), s["m"].astype(int), s["G0"], s["J"].double()
        goff, loff = s["goff"].astype(int), s["loff"].astype(int)
        lam = torch.empty(int(n.sum()), device="cuda", dtype=torch.float64)
        for k in np.unique(n):
            at = np.flatnonzero(n == k)
            mk = int(m[at[0]])
            X = torch.stack([G[goff[i]: goff[i] + mk * k].view(k, mk).T for i in at])
            Jk = torch.stack([J[loff[i]: loff[i] + k] for i in at])
            w = torch.linalg.eigvalsh((X * Jk[:, None, :]) @ X.mT)
            if mk > k:
                keep = torch.sort(torch.argsort(w.abs(), dim=1, descending=True)[:, :k], dim=1)[0]
                w = torch.gather(w, 1, keep)
            for r, i in zip(w, at):
                lam[loff[i]: loff[i] + k] = r
        return dict(lam=lam, V=None) if s["v"] else dict(lam=lam)
    if case["kind"] == "train":
        G, w, C = s["G"], s["w"], s["C"]
        lam, U = torch.linalg.eigh(G @ G.mT)
        U_bar = torch.zeros_like(U)
        U_bar[:, :, -8:] = 2.0 * C @ (C.T @ U[:, :, -8:])
        H_bar = _adjoint(lam, U, w.expand_as(lam), U_bar)
        return dict(lam=lam, U=U * _phase(U), grad=2.0 * H_bar @ G)
    return dict(H_bar=_adjoint(s["lam"], s["U"], s["lam_bar"], s["U_bar"]))
