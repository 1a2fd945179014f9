"""Coarse solve by planes from both ends: every count of planes up to six (one plane, two without a plane before the
middle's partner, odd and even counts) against the dense inverse, to rounding (1e-12, the tolerance of the 48^3
comparison of the same two forms)."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines only
    pytest.skip("CUDA device required", allow_module_level=True)

import paper_1205_1926_gb300 as T  # noqa: E402


@pytest.mark.parametrize("n_planes", [1, 2, 3, 4, 5, 6])
def test_planes_equal_dense(n_planes):
    nz = 2 * n_planes
    w = W.Workload(name="pl", nel=(4, 3, nz), cuts=((0, 2, 4), (0, 3), tuple(range(0, nz + 1, 2))),
                   length=(1.0, 0.8, 1.5))
    outs = []
    for coarse in (T.COARSE_DENSE, T.COARSE_PLANES):
        ctx = T.Context(w, coarse=coarse)
        y = torch.zeros(ctx.sizes["n_mult"], dtype=torch.float64, device="cuda")
        ctx.apply("projector", torch.as_tensor(W.seeded_vector(ctx.sizes["n_mult"], seed=7), device="cuda"), y)
        outs.append(y.cpu().numpy())
        ctx.close()
    assert np.linalg.norm(outs[1] - outs[0]) <= 1e-12 * np.linalg.norm(outs[0])
