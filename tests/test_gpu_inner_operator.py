"""GPU test of the inner operator (CG on S D~^-1, the correction mapped back
by D~^-1) over the Moebius coefficients its recurrences take: Shamir (c = 0),
c / b near 1 and negative, both chiralities of the shift, no shift, every
compiled Ls, every storage precision.  The oracle's operator judges each
solution at the solver's own target, 1e-10.
"""
import numpy as np
import pytest

from paper_1706_05843_gb300 import inputs as I

pytestmark = pytest.mark.gpu

CASES = [
    (4, dict(b=1.0, c=0.0, pm=1, beta=-1.0)),
    (8, dict(b=1.0, c=0.9, pm=-1, beta=0.7)),
    (12, dict(b=1.2, c=-0.2, pm=1, beta=0.5)),
    (16, dict(b=1.5, c=0.5, pm=-1, beta=0.0)),
    (12, dict(b=2.0, c=1.0, pm=1, beta=-1.0)),
]


@pytest.mark.parametrize("Ls,kw", CASES)
@pytest.mark.parametrize("inner", ["f64", "f32", "f16", "bf16"])
def test_solution_judged_by_the_oracle(Ls, kw, inner):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle as O
    from paper_1706_05843_gb300 import binding as B
    from paper_1706_05843_gb300 import build
    build.build()
    O.build()
    dims = (4, 2, 4, 6)
    act = dict(M5=1.8, m1=0.1, m2=1.0, m3=0.2, t_bc=-1, **kw)
    U = I.gauge_field(dims, 0.5, 3)
    phi = I.gaussian_fermion(dims, Ls, 1001)
    o = O.Oracle(O.Action(dims=dims, Ls=Ls, **act), U)
    s = B.Solver(U, dims, Ls, **act)
    x = torch.from_numpy(phi).cuda()
    for form, op in ((0, o.hsys), (1, o.k)):
        sol, st = s.solve(x, tol=1e-10, inner=inner, rhs_form=form)
        r = np.linalg.norm(phi - op(sol.cpu().numpy())) / np.linalg.norm(phi)
        assert r <= 1e-10 * (1 + 1e-3), (form, r, st.inner_iters)
    s.close()


@pytest.mark.parametrize("inner", ["f64", "f32"])
@pytest.mark.parametrize("seed", [1001, 1002, 1003, 1004])
def test_last_step_leaves_room(inner, seed):
    """The last inner solve aims 5% below the tolerance, so that neither the
    FP64 residual nor the full-lattice check lands just above it (FP32
    recurrence against FP64 residual: about 1e-3, bound 2%); also for the
    chirality whose shift makes the system nearly singular."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1706_05843_gb300 import binding as B
    from paper_1706_05843_gb300 import build
    build.build()
    dims, Ls = (4, 4, 4, 6), 8
    act = dict(M5=1.8, b=1.5, c=0.5, m1=0.08, m2=1.0, m3=0.08, beta=-1.0, t_bc=-1)
    U = I.gauge_field(dims, 0.6, seed)
    x = torch.from_numpy(I.gaussian_fermion(dims, Ls, seed)).cuda()
    for pm in (1, -1):
        s = B.Solver(U, dims, Ls, pm=pm, **act)
        _, st = s.solve(x, tol=1e-12, inner=inner)
        _, (sb,) = B.solve_batched([s], [x], tol=1e-12, inner=inner)
        s.close()
        assert st.true_res <= 0.97e-12 and sb.true_res <= 0.97e-12, (pm, st.true_res, sb.true_res)
