"""GPU test of the hop statistics of a plain FP64 solve: the launches sampled
inside the solver's graph and those timed one by one (kernel_timing) cover the
same work, the input pass of the two even-to-odd halves included.

The pass is 5 to 7% of the four launches' time at this size; the events of
either mode add a microsecond or two to 290, and repeated runs of one mode
differ by less than 1%: 3% separates the two.  The solves stop at their
iteration cap, so that no launch returns early on a finished solve.
"""
import pytest

from paper_1706_05843_gb300 import inputs as I

pytestmark = pytest.mark.gpu

ACT = dict(M5=1.8, b=1.5, c=0.5, m1=0.04, m2=1.0, m3=0.04, beta=-1.0, pm=1, t_bc=-1)


def test_both_modes_time_the_same_work():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1706_05843_gb300 import build
    build.build()
    from paper_1706_05843_gb300 import binding as B
    dims, Ls = (16, 16, 16, 16), 16
    s = B.Solver(I.gauge_field(dims, 0.3, 1), dims, Ls, **ACT)
    rhs = torch.view_as_complex(torch.randn(16, 16, 16, 16, Ls, 4, 3, 2, dtype=torch.float64, device="cuda"))
    ms, per = {0: [], 1: []}, {}
    for timing in (0, 1, 0, 1, 0, 1, 0, 1):
        _, st = s.solve(rhs, tol=1e-14, inner="f64", max_iter=32, max_outer=1, check=False, kernel_timing=timing)
        ms[timing].append(st.hop_ms / st.hop_launches)
        per[timing] = st.hop_bytes / st.hop_launches
    s.close()
    a, b = (sorted(ms[t][1:])[1] for t in (0, 1))  # medians after a warm-up
    print(f"graph {a * 1e3:.1f} us, one by one {b * 1e3:.1f} us a launch")
    assert abs(a - b) <= 0.03 * a
    assert per[1] == pytest.approx(per[0], rel=1e-12)
