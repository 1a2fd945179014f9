"""F x = B K^+ B^T x by the boundary form of the digit product against B, B^T and the full form, at several scales of x.

Each form is off by at most 4 n 2^-54 max|x_box| max_j |K^+_ij| in entry i (both operands are rounded to 55 bits below their
row's largest entry); a row of B adds its entries' bounds, and the sums over it round to 8 x 2^-53 of their terms.  The
bound is linear in x, as the error is.
"""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines only
    pytest.skip("CUDA device required", allow_module_level=True)

import paper_1205_1926_gb300 as T  # noqa: E402


@pytest.mark.parametrize("scale", [1e-6, 1.0, 1e6])
def test_boundary_form(scale):
    a, parts = (5, 4, 3), (3, 2, 2)
    w = W.Workload(name="boxes", nel=tuple(x * p for x, p in zip(a, parts)),
                   cuts=tuple(tuple(x * i for i in range(p + 1)) for x, p in zip(a, parts)))
    ctx = T.Context(w)
    nd, m, ns = (ctx.sizes[k] for k in ("n_dof", "n_mult", "n_sub"))
    n = nd // ns
    dev = lambda v: torch.as_tensor(np.ascontiguousarray(v), device="cuda")  # noqa: E731
    z = torch.zeros(nd, dtype=torch.float64, device="cuda")
    ctx.assemble_tangent(z, z)
    y, v = torch.zeros(m, dtype=torch.float64, device="cuda"), torch.zeros_like(z)
    kmax = np.zeros(n)                  # largest entry of each row of K^+, from unit vectors
    for j0 in range(0, n, ns):
        x = np.zeros(nd)
        for p in range(min(ns, n - j0)):
            x[p * n + j0 + p] = 1.0
        ctx.apply("kdag", dev(x), v)
        h = np.abs(v.cpu().numpy().reshape(ns, n)[:min(ns, n - j0)])
        kmax = np.maximum(kmax, h.max(axis=0))
    rows, cols, vals = T.Plan(w).export_B()
    x = scale * np.random.default_rng(7).standard_normal(m)
    bt = np.zeros(nd)
    np.add.at(bt, cols, vals * x[rows])
    ctx.apply("F", dev(x), y)
    ctx.apply("kdag", dev(bt), v)
    full = v.cpu().numpy()
    ref, tol = np.zeros(m), np.zeros(m)
    np.add.at(ref, rows, vals * full[cols])
    largest = np.abs(bt).reshape(ns, n).max(axis=1)
    entry = 2 * 4.0 * n * 2.0 ** -54 * np.repeat(largest, n) * np.tile(kmax, ns) + 8 * 2.0 ** -53 * np.abs(full)
    np.add.at(tol, rows, np.abs(vals) * entry[cols])
    assert (np.abs(y.cpu().numpy() - ref) <= tol).all()
