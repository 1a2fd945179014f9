"""Return mapping of pure shear states over the whole exponent range, against extended precision.

With no increment tau = (0, 0, 0, s, 0, 0) is deviatoric, |dev tau| = sqrt(2) s, and the result follows in closed form:
Phi = sqrt(3) s - (sigma_y + H kappa), d kappa = Phi / (3 mu + H), d sigma = -(3 mu / (3 mu + H)) Phi / sqrt(3) in the xy
entry.  Bounds: eight FP64 roundings of the magnitudes that enter (sqrt(3) s + yield), 8 x 2^-53 of them.
"""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines only
    pytest.skip("CUDA device required", allow_module_level=True)

import paper_1205_1926_gb300 as T  # noqa: E402


def shear_states(n, seed, sigma_y, hardening):
    """Magnitudes from 1e-300 to 1e150, many close to yield, and the special values."""
    rng = np.random.default_rng(seed)
    s, kap = 10.0 ** rng.uniform(-300.0, 150.0, n), 1e-3 * rng.random(n)
    near = slice(0, n // 2)
    s[near] = (sigma_y + hardening * kap[near]) / np.sqrt(3.0) * (
        1.0 + rng.choice((-0.5, 1.0), n // 2) * 10.0 ** rng.uniform(-9, 0, n // 2))
    s[n // 2:n // 2 + 40] = 10.0 ** rng.uniform(-2, 12, 40)
    s[-4:] = 0.0, np.inf, np.nan, 1e200            # 1e200: the square overflows
    s *= rng.choice((-1.0, 1.0), n)
    return s, kap


@pytest.mark.parametrize("seed", [1, 2])
def test_pure_shear(seed):
    w = W.SMALL4
    ctx = T.Context(w)
    n, ng = ctx.sizes["n_dof"], ctx.sizes["n_gp"]
    mat = w.material
    mu, H, sigma_y = mat["young"] / (2.0 * (1.0 + mat["poisson"])), mat["hardening"], mat["sigma_y"]
    s, kap = shear_states(ng, seed, sigma_y, H)
    sig = np.zeros((6, ng))
    sig[3] = s
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    ctx.set_state(sigma=dev(sig), kappa=dev(kap))
    ds, dk = torch.zeros(6, ng, dtype=torch.float64, device="cuda"), torch.zeros(ng, dtype=torch.float64, device="cuda")
    pl = torch.zeros(ng, dtype=torch.uint8, device="cuda")
    ctx.return_map(dev(np.zeros(n)), ds, dk, pl)
    ds, dk, pl = ds.cpu().numpy(), dk.cpu().numpy(), pl.cpu().numpy()
    L = np.longdouble
    fine = np.isfinite(s) & (np.abs(s) < 1e150)
    y = L(sigma_y) + L(H) * kap.astype(L)
    phi = np.sqrt(L(3)) * np.abs(s[fine].astype(L)) - y[fine]
    yields = phi > 1e-12 * y[fine]
    assert yields.any() and not yields.all()
    assert np.array_equal(pl[fine] != 0, yields)
    phi = np.where(yields, phi, 0)
    c = 3 * L(mu) / (3 * L(mu) + L(H))
    tol = 8 * 2.0 ** -53 * (np.sqrt(3.0) * np.abs(s[fine]) + y[fine].astype(float))
    ref_k = (phi / (3 * L(mu) + L(H))).astype(float)
    assert np.all(np.abs(dk[fine] - ref_k) <= tol / (3 * mu + H))
    ref_s = (-np.sign(s[fine]) * c * phi / np.sqrt(L(3))).astype(float)
    assert np.all(np.abs(ds[3][fine] - ref_s) <= tol)
    for q in (0, 1, 2, 4, 5):
        assert np.all(ds[q][fine] == 0.0)
    assert pl[-3] == 1 and pl[-1] == 1 and pl[-2] == 0   # infinite and overflowing: beyond yield; not a number: not
    assert not np.isfinite(ds[3][-3])
