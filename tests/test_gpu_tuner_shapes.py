"""GPU tests of what the autotuner shares between contexts: timings of the same
lattice only, and of the same boundary conditions."""
import numpy as np
import pytest

from paper_1706_05843_gb300 import inputs as I

pytestmark = pytest.mark.gpu

ACT = dict(M5=1.8, b=1.5, c=0.5, m1=0.04, m2=1.0, m3=0.04, beta=-1.0, pm=1, t_bc=-1)


def tuned(B, torch, dims, Ls, gparity=0):
    """The launch times that a context of this lattice reports after an FP32 solve (4 kinds, 4 variants, 2 precisions)."""
    s = B.Solver(I.gauge_field(dims, 0.3, 1), dims, Ls, gparity=gparity, **ACT)
    x = I.gaussian_fermion(dims, Ls, 7)
    x = np.stack([x, x]) if gparity else x
    sol, st = s.solve(torch.from_numpy(x).cuda(), tol=1e-8, inner="f32")
    t = [B.lib().eofa_tile_time(s.ctx, p, k, v) for p in (0, 1) for k in range(4) for v in range(4)]
    assert st.true_res <= 1e-8
    s.close()
    return t


def test_timings_belong_to_one_lattice():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1706_05843_gb300 import build
    build.build()
    from paper_1706_05843_gb300 import binding as B
    a = tuned(B, torch, (4, 12, 2, 8), 8)
    assert tuned(B, torch, (4, 12, 2, 8), 8) == a         # the same lattice: from the cache
    assert tuned(B, torch, (12, 4, 2, 8), 8) != a         # same X Y
    assert tuned(B, torch, (4, 12, 8, 2), 8) != a         # same Z T
    b = tuned(B, torch, (4, 12, 2, 4), 8, gparity=1)      # two flavours stacked along t: X x Y x Z x 2 T
    assert b != a
    assert tuned(B, torch, (4, 12, 2, 4), 8, gparity=2) != b
