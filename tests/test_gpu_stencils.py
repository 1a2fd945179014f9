"""K x and the band of K from the assembled stencils: boxes one and more elements thick, unequal element edges,
elastic and partly yielding, against the oracle (1e-11 of the largest entry, as the operator parity tests)."""
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


@pytest.mark.parametrize("nel,cuts", [
    ((1, 1, 2), ((0, 1), (0, 1), (0, 2))),
    ((3, 1, 4), ((0, 1, 3), (0, 1), (0, 4))),
    ((5, 4, 6), ((0, 2, 5), (0, 1, 4), (0, 3, 6))),
])
@pytest.mark.parametrize("hot", [0, 1, 8])
def test_apply_K(nel, cuts, hot):
    import scipy.sparse as sp
    w = W.Workload(name="st", nel=nel, cuts=cuts, length=(1.0, 0.7, 1.3))
    m = ElastoplasticModel(w)
    du, _ = W.seeded_partly_plastic_increment(w, 5, hot)
    if not hot:
        du = 0.0 * du
    ctx = T.Context(w)
    n = ctx.sizes["n_dof"]
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    ctx.assemble_tangent(dev(du), dev(np.zeros(n)))
    Kb, _, _ = m.assemble(du, np.zeros(n))
    x = W.seeded_vector(n, 6)
    y = torch.zeros(n, dtype=torch.float64, device="cuda")
    ctx.apply("K", dev(x), y)
    ref = sp.block_diag(Kb) @ x
    assert np.abs(y.cpu().numpy() - ref).max() <= 1e-11 * np.abs(ref).max()
    ctx.apply("kdag", dev(x), y)
    ref = np.concatenate([FixingNodeInverse(K, s.fixing_dofs()).apply(x[m.dec.dof_off[p]:m.dec.dof_off[p + 1]])
                          for p, (K, s) in enumerate(zip(Kb, m.dec.subs))])
    assert np.linalg.norm(y.cpu().numpy() - ref) <= 1e-10 * np.linalg.norm(ref)


@pytest.mark.parametrize("nel,cuts", [
    ((4, 4, 4), ((0, 2, 4), (0, 2, 4), (0, 4))),      # free faces: node boxes with and without them
    ((3, 5, 4), ((0, 1, 3), (0, 5), (0, 1, 2, 4))),   # boxes one element thick: no unconstrained node in some
    ((8, 8, 4), ((0, 8), (0, 4, 8), (0, 4))),
])
@pytest.mark.parametrize("hot", [0, 1])
def test_dirichlet_preconditioner_on_node_boxes(nel, cuts, hot):
    """Bbar Sbar Bbar^T x through the K_ii of the unconstrained nodes, elastic and partly yielding (1e-11 of the
    largest entry)."""
    from oracle.tfeti import TFETISolver
    w = W.Workload(name="di", nel=nel, cuts=cuts)
    m = ElastoplasticModel(w)
    du, _ = W.seeded_partly_plastic_increment(w, 9, hot)
    if not hot:
        du = 0.0 * du
    ctx = T.Context(w, precond=T.PRECOND_DIRICHLET)
    n, nm = ctx.sizes["n_dof"], ctx.sizes["n_mult"]
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    ctx.assemble_tangent(dev(du), dev(np.zeros(n)))
    Kb, _, _ = m.assemble(du, np.zeros(n))
    sol = TFETISolver(m.dec, Kb, [FixingNodeInverse(K, s.fixing_dofs()) for K, s in zip(Kb, m.dec.subs)],
                      precond="dirichlet")
    x = W.seeded_vector(nm, 8)
    y = torch.zeros(nm, dtype=torch.float64, device="cuda")
    ctx.apply("precond", dev(x), y)
    ref = sol.apply_precond(x)
    assert np.abs(y.cpu().numpy() - ref).max() <= 1e-11 * np.abs(ref).max()
