"""GPU test of the operator applications on lattices where one grid serves both
parities and a CTA walks several blocks of sites: the double-buffered links,
the reuse of the column tiles and of the staged y, canonical stores of a last
block that is not full (Ls = 4).  Against the FP64 oracle; the norm bound is
that of the small lattices (test_gpu_fixed_hop).
"""
import numpy as np
import pytest

from paper_1706_05843_gb300 import inputs as I

pytestmark = pytest.mark.gpu

ACT = dict(M5=1.8, b=1.5, c=0.5, m1=0.04, m2=1.0, m3=0.04, beta=-1.0, pm=1, t_bc=-1)


@pytest.mark.parametrize("dims,Ls,pm", [
    ((12, 12, 12, 16), 12, -1),  # column phase for K^dag
    ((12, 12, 12, 10), 16, 1),   # shuffles
    ((10, 10, 10, 12), 8, 1),
    ((6, 10, 14, 18), 4, -1),    # 7560 sites a parity, 16 a block: the last one half full
])
def test_middle_sizes(dims, Ls, pm):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1706_05843_gb300 import build
    build.build()
    from paper_1706_05843_gb300 import binding as B
    import oracle as O
    O.build()
    act = dict(ACT, pm=pm)
    U, x = I.gauge_field(dims, 0.5, 3), I.gaussian_fermion(dims, Ls, 1001)
    o = O.Oracle(O.Action(dims=dims, Ls=Ls, **act), U)
    s = B.Solver(U, dims, Ls, **act)
    xt = torch.from_numpy(x).cuda()
    for f, ref in ((B.eofa_apply, o.k), (B.eofa_apply_dag, lambda v: o.k(v, dag=True)), (B.eofa_apply_h, o.hsys)):
        out = torch.full_like(xt, float("nan"))
        f(s.ctx, xt, out)
        r = ref(x)
        assert np.linalg.norm(out.cpu().numpy() - r) <= 1e-14 * np.linalg.norm(r)
    s.close()
