"""Tensor-core FP64 products with a shape's dense K^+ (digit splitting): accuracy of the product itself.

K^+ of a box is read column by column through unit vectors; the product with a random, constant or badly scaled
x is then compared with the sum of those columns in extended precision.  Both operands are rounded to 55 bits
below the power of two above their row's largest entry (2^-55 of it at most), the columns were read with the
same rounding, and the FP64 rounding of the result is 2^-53: with n terms the entry i is off by at most
4 n 2^-54 max|x| max_j |K^+_ij|.
"""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines only
    pytest.skip("CUDA device required", allow_module_level=True)

import paper_1205_1926_gb300 as T  # noqa: E402


def boxes(a, parts=(2, 2, 2)):
    """parts boxes of a = (ax, ay, az) elements each."""
    return W.Workload(name="boxes", nel=tuple(x * p for x, p in zip(a, parts)),
                      cuts=tuple(tuple(x * i for i in range(p + 1)) for x, p in zip(a, parts)))


def dev(x):
    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


# tiles of 64 output dofs with remainders of 17 (81), 52 (180), 32 (288) and 5 (1029), K below and above the
# chunks of 192 with odd numbers of 16-column stages (81, 1029), and 130 boxes (two tiles of 128 rows)
@pytest.mark.parametrize("a,parts", [((2, 2, 2), (2, 2, 2)), ((4, 3, 2), (2, 2, 1)), ((5, 3, 3), (2, 2, 2)),
                                     ((6, 6, 6), (2, 2, 2)), ((2, 2, 2), (13, 5, 2))])
def test_product_against_extended_precision(a, parts):
    w = boxes(a, parts)
    ctx = T.Context(w)
    nd, ns = ctx.sizes["n_dof"], ctx.sizes["n_sub"]
    n = nd // ns
    ctx.assemble_tangent(torch.zeros(nd, dtype=torch.float64, device="cuda"),
                         torch.zeros(nd, dtype=torch.float64, device="cuda"))
    y = torch.zeros(nd, dtype=torch.float64, device="cuda")
    cols = np.empty((n, n))
    for j0 in range(0, n, ns):          # one unit vector per box and call
        x = np.zeros(nd)
        for p in range(min(ns, n - j0)):
            x[p * n + j0 + p] = 1.0
        ctx.apply("kdag", dev(x), y)
        h = y.cpu().numpy().reshape(ns, n)
        for p in range(min(ns, n - j0)):
            cols[:, j0 + p] = h[p]
    rng = np.random.default_rng(5)
    X = rng.standard_normal((ns, n))
    X[1] = 1.0                          # every digit product of one sign
    X[2] *= np.exp(12.0 * rng.standard_normal(n))
    X[3] = 0.0
    ctx.apply("kdag", dev(X.ravel()), y)
    got = y.cpu().numpy().reshape(ns, n)
    fixed = ~cols.any(axis=0)           # the six fixing dofs: zero rows and columns
    assert fixed.sum() == 6 and not got[:, fixed].any()
    kmax = np.abs(cols).max(axis=1)
    for p in (0, 1, 2, 3, ns - 1):
        ref = (cols.astype(np.longdouble) * X[p].astype(np.longdouble)).sum(axis=1)
        tol = 4.0 * n * 2.0 ** -54 * np.abs(X[p][~fixed]).max() * kmax
        assert (np.abs(got[p] - ref) <= tol).all()


def test_boundary_form_is_the_full_form():
    """F x = B K^+ B^T x: the product over the boundary dofs against the full product, same bound as above."""
    w = boxes((5, 4, 3), (3, 2, 2))
    ctx = T.Context(w)
    nd, m = ctx.sizes["n_dof"], ctx.sizes["n_mult"]
    z = torch.zeros(nd, dtype=torch.float64, device="cuda")
    ctx.assemble_tangent(z, z)
    rows, cols, vals = T.Plan(w).export_B()
    x = np.random.default_rng(7).standard_normal(m)
    bt = np.zeros(nd)
    np.add.at(bt, cols, vals * x[rows])
    y, v = torch.zeros(m, dtype=torch.float64, device="cuda"), torch.zeros_like(z)
    ctx.apply("F", dev(x), y)
    ctx.apply("kdag", dev(bt), v)
    ref = np.zeros(m)
    np.add.at(ref, rows, vals * v.cpu().numpy()[cols])
    n = nd // ctx.sizes["n_sub"]
    assert np.abs(y.cpu().numpy() - ref).max() <= 8.0 * n * 2.0 ** -54 * np.abs(bt).max() * 8 * np.abs(ref).max()


def test_non_finite_input_stays_in_its_box():
    w = boxes((3, 3, 3))
    ctx = T.Context(w)
    nd, ns = ctx.sizes["n_dof"], ctx.sizes["n_sub"]
    n = nd // ns
    z = torch.zeros(nd, dtype=torch.float64, device="cuda")
    ctx.assemble_tangent(z, z)
    x = np.random.default_rng(9).standard_normal((ns, n))
    ref, y = torch.zeros_like(z), torch.zeros_like(z)
    ctx.apply("kdag", dev(x.ravel()), ref)
    for bad in (np.nan, np.inf):
        x[2, n // 2] = bad
        ctx.apply("kdag", dev(x.ravel()), y)
        got, want = y.cpu().numpy().reshape(ns, n), ref.cpu().numpy().reshape(ns, n)
        keep = [p for p in range(ns) if p != 2]
        assert np.array_equal(got[keep], want[keep])
        free = want[2] != 0.0
        assert np.isnan(got[2][free]).all()
