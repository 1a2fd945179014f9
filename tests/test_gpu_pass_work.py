"""Work of the FP64 K^+ passes as launched: digit products of the boxes on their shape's factor, in the boundary or the
full form, and banded sweeps of the others, by direct count."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines only
    pytest.skip("CUDA device required", allow_module_level=True)

import paper_1205_1926_gb300 as T  # noqa: E402


@pytest.mark.parametrize("hot", [0, 3, 8])
def test_counted_passes(hot):
    cuts = (0, 4, 8)
    w = W.Workload(name="work", nel=(8, 8, 8), cuts=(cuts, cuts, cuts))     # 8 boxes of 375 dofs, 98 boundary nodes
    ctx = T.Context(w)
    nd, m = ctx.sizes["n_dof"], ctx.sizes["n_mult"]
    du, _ = W.seeded_partly_plastic_increment(w, 3, hot)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    zero = torch.zeros(nd, dtype=torch.float64, device="cuda")
    ctx.assemble_tangent(dev(du if hot else 0.0 * du), zero)
    x, y = dev(W.seeded_vector(m, 1)), torch.zeros(m, dtype=torch.float64, device="cuda")
    f, u = torch.zeros_like(zero), torch.zeros_like(zero)
    ctx.traction_load((1.0, 0.0, 0.0), f)
    n, n_bd, bw, nb = 375, 3 * 98, 3 * (25 + 5 + 1) + 2, 32
    nblk = -(-n // nb)
    banded = hot * 4.0 * (nblk * nb * bw + nblk * nb * (nb + 1) / 2.0)
    ctx.timing_reset(True)
    for _ in range(3):
        ctx.apply("F", x, y)
    got = ctx.pass_work()
    assert got == {"passes": 3, "banded_passes": 3 if hot else 0, "digit_flops": 3 * 56.0 * (8 - hot) * n_bd ** 2,
                   "banded_flops": 3 * banded}
    ctx.timing_reset(True)
    info = ctx.dual_pcg(f, u, rtol=1e-8)
    got = ctx.pass_work()
    full = got["passes"] - info["iterations"]           # residual passes need all dofs, F-applies the boundary
    assert full >= 1 and got["passes"] == info["f_applies"]
    assert got["digit_flops"] == 56.0 * (8 - hot) * (info["iterations"] * n_bd ** 2 + full * n ** 2)
    assert got["banded_flops"] == got["passes"] * banded
    ctx.timing_reset(False)
    assert ctx.pass_work()["digit_flops"] == 0.0
