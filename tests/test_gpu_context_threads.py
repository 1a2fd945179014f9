"""Contexts of several host threads whose kernels need different amounts of shared memory do not undercut each other.

Six threads assemble tangents with Woodbury corrections of many and of few plastic points per box (the substitution's
shared memory goes with the largest count); no call may fail, and each thread's K^+ apply stays what it is alone.
"""
import threading

import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines only
    pytest.skip("CUDA device required", allow_module_level=True)

import paper_1205_1926_gb300 as T  # noqa: E402


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def increment(ctx, w, lo, hi):
    """A seeded increment whose largest count of plastic points in a box lies in [lo, hi]."""
    n, ng, ns = ctx.sizes["n_dof"], ctx.sizes["n_gp"], ctx.sizes["n_sub"]
    out = [torch.zeros(6, ng, dtype=torch.float64, device="cuda"), torch.zeros(ng, dtype=torch.float64, device="cuda"),
           torch.zeros(ng, dtype=torch.uint8, device="cuda")]
    for s in np.geomspace(2e-4, 1.2e-3, 60):
        du, _ = W.seeded_partly_plastic_increment(w, 3, ns, hot_scale=s)
        ctx.return_map(dev(du), *out)
        most = int(out[2].cpu().numpy().reshape(ns, -1).sum(axis=1).max())
        if lo <= most <= hi:
            return dev(du)
    raise AssertionError("no such increment")


def test_woodbury_sizes_in_several_threads():
    cuts = (0, 4, 8)
    w = W.Workload(name="threads", nel=(8, 8, 8), cuts=(cuts, cuts, cuts))
    ctxs, dus = [], []
    for lo, hi in 3 * ((70, 96), (1, 12)):
        ctx = T.Context(w, stream=torch.cuda.Stream())
        ctx.set_precision(True, 1e-4)
        ctxs.append(ctx)
        dus.append(increment(ctx, w, lo, hi))
    n = ctxs[0].sizes["n_dof"]
    zero, x = torch.zeros(n, dtype=torch.float64, device="cuda"), dev(W.seeded_vector(n, 1))
    torch.cuda.synchronize()
    alone = []
    for ctx, du in zip(ctxs, dus):
        before = ctx.woodbury_stats()["subdomains"]
        y = torch.zeros_like(zero)
        torch.cuda.synchronize()
        ctx.assemble_tangent(du, zero)
        ctx.apply("kdag", x, y)
        assert ctx.woodbury_stats()["subdomains"] > before
        alone.append(y)
    errors = []

    def work(k):
        try:
            for _ in range(600):
                ctxs[k].assemble_tangent(dus[k], zero)
        except T.TfetiError as e:
            errors.append((k, str(e)))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(ctxs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for ctx, ref in zip(ctxs, alone):
        y = torch.zeros_like(zero)
        torch.cuda.synchronize()
        ctx.apply("kdag", x, y)
        assert torch.equal(y, ref)
