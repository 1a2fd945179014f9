"""K^+ applies of boxes with factors of their own by clusters of CTAs, against the oracle's factors.

Few boxes yield, so each gets the most CTAs its row blocks allow; box sizes give full and ragged last blocks,
half bandwidths below and above the window's powers of two, and 32- and 16-row blocks.  Tolerance: that of the
K^+ parity tests (1e-10 relative; FP32: 1e-5).
"""
import numpy as np
import pytest

import workloads as W
from oracle.decomp import FixingNodeInverse
from oracle.ssn import ElastoplasticModel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines only
    pytest.skip("CUDA device required", allow_module_level=True)

import paper_1205_1926_gb300 as T  # noqa: E402


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def work(nel, cuts):
    return W.Workload(name="cl", nel=nel, cuts=cuts)


# dofs 27 x 3 = 81 (three blocks, the last of 17 rows), 144, 192 (exact), 375; two shapes side by side; boxes
# large enough for 16-row blocks beside small ones (10^3 elements: 3993 dofs)
@pytest.mark.parametrize("w,hot", [
    (work((4, 4, 4), ((0, 2, 4),) * 3), 8),
    (work((6, 3, 5), ((0, 3, 6), (0, 3), (0, 2, 5))), 3),
    (work((6, 6, 3), ((0, 3, 6), (0, 3, 6), (0, 3))), 2),
    (work((4, 8, 8), ((0, 4), (0, 4, 8), (0, 4, 8))), 1),
    (work((10, 10, 14), ((0, 10), (0, 10), (0, 10, 14))), 2),
])
def test_own_factor_boxes_against_oracle(w, hot):
    m = ElastoplasticModel(w)
    du, boxes = W.seeded_partly_plastic_increment(w, 3, hot)
    ctx = T.Context(w)
    n, nm = ctx.sizes["n_dof"], ctx.sizes["n_mult"]
    zero = np.zeros(n)
    ctx.assemble_tangent(dev(du), dev(zero))
    Kb, _, _ = m.assemble(du, zero)
    inv = [FixingNodeInverse(K, s.fixing_dofs()) for K, s in zip(Kb, m.dec.subs)]

    def kdag(x):
        return np.concatenate([inv[p].apply(x[m.dec.dof_off[p]:m.dec.dof_off[p + 1]]) for p in range(len(inv))])

    rng = np.random.default_rng(4)
    x, lam = rng.standard_normal(n), rng.standard_normal(nm)
    y, f = torch.zeros(n, dtype=torch.float64, device="cuda"), torch.zeros(nm, dtype=torch.float64, device="cuda")
    ctx.apply("kdag", dev(x), y)
    ref = kdag(x)
    for p in range(len(inv)):
        s = slice(m.dec.dof_off[p], m.dec.dof_off[p + 1])
        assert np.linalg.norm(y.cpu().numpy()[s] - ref[s]) <= 1e-10 * np.linalg.norm(ref[s])
    ctx.apply("F", dev(lam), f)
    fref = m.dec.B @ kdag(m.dec.B.T @ lam)
    assert np.linalg.norm(f.cpu().numpy() - fref) <= 1e-10 * np.linalg.norm(fref)
    g, dlam = torch.zeros_like(f), dev(lam)
    for _ in range(200):                # repeated applies are bitwise equal
        ctx.apply("F", dlam, g)
        assert torch.equal(f, g)
    ctx.set_precision(True, 1e-4)
    ctx.set_woodbury(0)
    ctx.assemble_tangent(dev(du), dev(zero))
    ctx.apply("F32", dev(lam), g)
    assert np.linalg.norm(g.cpu().numpy() - fref) <= 1e-5 * np.linalg.norm(fref)
