"""Four load directions at once on the 48^3 cube in mixed precision with the history start, against the record of the
same run at commit 04c42b2 (tests/golden/cube48_mixed_ramp_record.json, written by running this file there).

The loads are multiples of the first-yield traction that the mixed solve itself gives, so a solve that ends with a
larger error within the same stopping tolerance (1e-11) shows in the plastic strains, which a few points just beyond
yield amplify some hundredfold.  Bounds: 1e-9 of the record in the 2-norm and 4e-8 at a point (over the larger of its value
and the root mean square), and the same points yield.
"""
import json
import os

import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines only
    pytest.skip("CUDA device required", allow_module_level=True)

import paper_1205_1926_gb300 as T  # noqa: E402

RECORD = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "cube48_mixed_ramp_record.json")


def plastic_strains(rec):
    cuts = tuple(range(0, 49, 8))
    w = W.Workload(name="ramp", nel=(48, 48, 48), cuts=(cuts, cuts, cuts))
    ctxs, loads = [], []
    for c in rec["cases"]:
        ctxs.append(T.Context(w, stream=torch.cuda.Stream()))
        ctxs[-1].set_precision(True, rec["inner_rtol"])
    n_dof, n_gp = ctxs[0].sizes["n_dof"], ctxs[0].sizes["n_gp"]
    for c in rec["cases"]:
        t_y = ctxs[0].first_yield_traction(c["direction"], rec["pcg_rtol"])
        f = torch.zeros(n_dof, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        ctxs[0].traction_load(tuple(c["factor"] * t_y * v for v in c["direction"]), f)
        torch.cuda.synchronize()
        loads.append(f / rec["steps"])
    torch.cuda.synchronize()
    for ctx in ctxs:
        ctx.set_recycling(rec["history"])
    for _ in range(rec["steps"]):
        T.time_step_cases(ctxs, loads, rec["newton_tol"], rec["pcg_rtol"])
    out = []
    for ctx in ctxs:
        kap = torch.zeros(n_gp, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        ctx.get_state(kappa=kap)
        out.append(kap.cpu().numpy())
        ctx.close()
    return out


def test_plastic_strains_as_recorded():
    with open(RECORD) as fh:
        rec = json.load(fh)
    for c, kap in zip(rec["cases"], plastic_strains(rec)):
        ref = np.zeros_like(kap)
        ref[c["points"]] = c["kappa"]
        assert np.array_equal(np.flatnonzero(kap), np.asarray(c["points"]))
        d, norm = np.abs(kap - ref), np.linalg.norm(ref)
        assert np.linalg.norm(d) <= 1e-9 * norm
        assert np.all(d <= 4e-8 * np.maximum(norm / np.sqrt(ref.size), np.abs(ref)))


if __name__ == "__main__":
    with open(RECORD) as fh:
        r = json.load(fh)
    for c, kap in zip(r["cases"], plastic_strains(r)):
        c["points"] = np.flatnonzero(kap).tolist()
        c["kappa"] = kap[c["points"]].tolist()
    with open(RECORD, "w") as fh:
        json.dump(r, fh)
