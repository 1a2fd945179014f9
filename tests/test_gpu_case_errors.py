"""A case context starts with a clear error word, whatever its recycled memory held."""
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines only
    pytest.skip("CUDA device required", allow_module_level=True)

import paper_1205_1926_gb300 as T  # noqa: E402


def test_case_context_in_recycled_memory():
    w = W.SMALL4
    base = T.Context(w)
    t_y = base.first_yield_traction(w.traction_dir)
    for _ in range(3):
        # fill a stretch of device memory with ones (also in small blocks) and give it back to the driver
        junk = [torch.full((k,), -1, dtype=torch.int32, device="cuda") for k in (1 << 24, *([64] * 2000))]
        torch.cuda.synchronize()
        del junk
        torch.cuda.empty_cache()
        case = T.Context.case_of(base, 450.0, 10000.0)
        df = torch.zeros(case.sizes["n_dof"], dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        case.traction_load(tuple(0.5 * t_y * c for c in w.traction_dir), df)
        assert case.time_step(df, 1e-8, 1e-10)["converged"]
        case.close()
