"""K^+ applies by clusters of CTAs on boxes of two and three row blocks, whose last block is solved right after its
forward rows have been exchanged: alternating right-hand sides, so that a value left over or arriving late from the
other solve shows as another result.  Repeated applies are bitwise equal, and as the oracle's (1e-10, the tolerance of
the K^+ parity tests)."""
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


# boxes of 36 dofs (a last block of 4 rows, one CTA's), 54 (22 rows) and 72 (three blocks, 8 rows)
@pytest.mark.parametrize("nel,cuts", [
    ((4, 1, 1), ((0, 2, 4), (0, 1), (0, 1))),
    ((4, 2, 1), ((0, 2, 4), (0, 2), (0, 1))),
    ((3, 2, 1), ((0, 3), (0, 2), (0, 1))),
    ((3, 2, 3), ((0, 3), (0, 2), (0, 1, 2, 3))),
])
def test_short_boxes_repeat_bitwise(nel, cuts):
    w = W.Workload(name="blk", nel=nel, cuts=cuts)
    m = ElastoplasticModel(w)
    du, _ = W.seeded_partly_plastic_increment(w, 3, 64)
    ctx = T.Context(w)
    n = ctx.sizes["n_dof"]
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    ctx.assemble_tangent(dev(du), dev(np.zeros(n)))
    Kb, _, _ = m.assemble(du, np.zeros(n))
    inv = [FixingNodeInverse(K, s.fixing_dofs()) for K, s in zip(Kb, m.dec.subs)]
    xs = [W.seeded_vector(n, 8), 1e6 * W.seeded_vector(n, 9)]
    first = []
    for x in xs:
        y = torch.zeros(n, dtype=torch.float64, device="cuda")
        ctx.apply("kdag", dev(x), y)
        for p in range(len(inv)):
            s = slice(m.dec.dof_off[p], m.dec.dof_off[p + 1])
            ref = inv[p].apply(x[s])
            assert np.linalg.norm(y.cpu().numpy()[s] - ref) <= 1e-10 * np.linalg.norm(ref)
        first.append(y)
    dx, y = [dev(x) for x in xs], torch.zeros_like(first[0])
    for k in range(2000):
        ctx.apply("kdag", dx[k % 2], y)
        assert torch.equal(y, first[k % 2])
