"""Every call that runs kernels with bounded waits reports one that gave up, and leaves nothing behind.

With the limit at 0 each wait of the banded solves and of the digit product gives up without a look; the kernels then
wait for their own copies as usual and end, so nothing is left pending.  The call returns TFETI_ERR_TIMEOUT, and with
the limit restored the same call gives the result it gave before, bit for bit.
"""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines only
    pytest.skip("CUDA device required", allow_module_level=True)

import paper_1205_1926_gb300 as T  # noqa: E402

TIMEOUT = 9


def cube(parts, a):
    c = tuple(range(0, parts * a + 1, a))
    return W.Workload(name="wait", nel=(parts * a,) * 3, cuts=(c, c, c))


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def new(n):
    return torch.zeros(n, dtype=torch.float64, device="cuda")


# eight boxes on their shape's digit product (hot 0) or by clusters with factors of their own (hot 8); two boxes of 24
# dofs by one CTA each; the Dirichlet preconditioner's solves
CASES = [(cube(2, 3), 0, T.PRECOND_LUMPED), (cube(2, 3), 8, T.PRECOND_LUMPED),
         (W.Workload(name="two", nel=(1, 1, 2), cuts=((0, 1), (0, 1), (0, 1, 2))), 0, T.PRECOND_LUMPED),
         (cube(2, 4), 0, T.PRECOND_DIRICHLET), (cube(2, 4), 3, T.PRECOND_DIRICHLET)]


@pytest.mark.parametrize("w,hot,precond", CASES)
@pytest.mark.parametrize("mixed", [False, True])
def test_each_call_reports_its_own(w, hot, precond, mixed):
    ctx = T.Context(w, precond=precond)
    n, m = ctx.sizes["n_dof"], ctx.sizes["n_mult"]
    if mixed:
        ctx.set_precision(True, 1e-4)
        ctx.set_woodbury(0)
        ctx.set_schur_threshold(1 << 20)   # F32 by banded sweeps
    du, _ = W.seeded_partly_plastic_increment(w, 3, hot)
    if not hot:
        du = 0.0 * du
    ctx.assemble_tangent(dev(du), new(n))
    x, lam, f = dev(W.seeded_vector(n, 1)), dev(W.seeded_vector(m, 2)), new(n)
    ctx.traction_load((1.0, 0.2, 0.3), f)
    calls = {"kdag": lambda out: ctx.apply("kdag", x, out), "F": lambda out: ctx.apply("F", lam, out),
             "solve": lambda out: ctx.dual_pcg(f, out, rtol=1e-10)}
    if precond == T.PRECOND_DIRICHLET:
        calls["precond"] = lambda out: ctx.apply("precond", lam, out)
    if mixed:
        calls["F32"] = lambda out: ctx.apply("F32", lam, out)
    size = {"kdag": n, "F": m, "solve": n, "precond": m, "F32": m}
    ref = {}
    for name, call in calls.items():
        ref[name] = new(size[name])
        call(ref[name])
    for name, call in calls.items():
        ctx.set_wait_limit(0)
        with pytest.raises(T.TfetiError) as e:
            call(new(size[name]))
        assert e.value.status == TIMEOUT, name
        ctx.set_wait_limit()
        out = new(size[name])
        call(out)                       # nothing of the call before is left to be blamed on this one
        assert torch.equal(out, ref[name]), name


def test_load_step_reports_and_recovers():
    w = cube(2, 4)
    ctx = T.Context(w)
    n = ctx.sizes["n_dof"]
    t = ctx.first_yield_traction(w.traction_dir)
    f, u0, u1 = new(n), new(n), new(n)
    ctx.traction_load(tuple(1.3 * t * c for c in w.traction_dir), f)
    ctx.set_wait_limit(0)
    with pytest.raises(T.TfetiError) as e:
        ctx.time_step(f, 1e-8, 1e-10)
    assert e.value.status == TIMEOUT
    with pytest.raises(T.TfetiError) as e:
        ctx.first_yield_traction(w.traction_dir)
    assert e.value.status == TIMEOUT
    ctx.set_wait_limit()
    assert ctx.time_step(f, 1e-8, 1e-10)["converged"]
    ctx.get_state(u=u0)
    other = T.Context(w)
    assert other.time_step(f, 1e-8, 1e-10)["converged"]
    other.get_state(u=u1)
    assert torch.equal(u0, u1)


def test_precision_change_reports_and_recovers():
    w = cube(2, 4)
    ctx, other = T.Context(w), T.Context(w)
    n = ctx.sizes["n_dof"]
    f, u0, u1 = new(n), new(n), new(n)
    ctx.traction_load((1.0, 0.2, 0.3), f)
    ctx.set_wait_limit(0)
    with pytest.raises(T.TfetiError) as e:
        ctx.set_precision(True, 1e-4)
    assert e.value.status == TIMEOUT
    ctx.set_wait_limit()
    for c, u in ((ctx, u0), (other, u1)):
        c.set_precision(True, 1e-4)
        c.set_schur_threshold(4)
        c.assemble_tangent(new(n), f)
        c.dual_pcg(f, u, rtol=1e-10)
    assert torch.equal(u0, u1)
    ctx.set_wait_limit(0)
    with pytest.raises(T.TfetiError) as e:
        ctx.set_schur_threshold(0)        # times the applies, banded ones among them
    assert e.value.status == TIMEOUT
    ctx.set_wait_limit()
    ctx.set_schur_threshold(4)
    ctx.dual_pcg(f, u1, rtol=1e-10)
    assert torch.equal(u0, u1)


def test_limits_refused():
    ctx = T.Context(cube(2, 2))
    for cycles in (-1, (1 << 31) + 1):
        with pytest.raises(T.TfetiError):
            ctx.set_wait_limit(cycles)
