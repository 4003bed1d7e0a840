"""GPU test of the tcgen05 convolution's walk at the edges of its cut: extents
of 1 and odd ones, a lattice within one tile and one that just exceeds it,
x in two and three blocks, one input slice per column and many, more columns
than one.  Reference and bound as in test_gpu_learned (the FP64 oracle with
BF16 rounding where the library stores BF16: only the order of the FP32 sums
differs, 1e-3; a misplaced tap, row or slot gives an error of order 1).
"""
import numpy as np
import pytest

from oracle import net as N

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,S", [
    ((1, 1, 1, 1), 1), ((2, 3, 1, 5), 2), ((5, 4, 3, 7), 3), ((66, 2, 2, 2), 1), ((130, 1, 2, 1), 2),
    ((16, 4, 2, 18), 1), ((6, 6, 4, 3), 7), ((4, 2, 2, 40), 90),
])
def test_net_forward_storage_model(dims, S):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1706_05843_gb300 import binding as B
    from paper_1706_05843_gb300 import build
    build.build()
    X, Y, Z, T = dims
    rng = np.random.default_rng(7)
    w = N.bf16_round(np.concatenate([rng.standard_normal(81 * co * ci) * np.sqrt(2.0 / (81 * ci))
                                     for ci, co in zip(N.CIN, N.COUT)]))
    x = N.bf16_round(rng.standard_normal((S, T, Z, Y, X, 24)))
    W = N.split(w)
    ref = N.conv(N.bf16_round(N.leaky(N.conv(N.bf16_round(N.leaky(N.conv(x, W[0]))), W[1]))), W[2])
    xt = torch.from_numpy(x.astype(np.float32)).cuda()
    out = torch.full_like(xt, float("nan"))
    B.eofa_net_forward(w.astype(np.float32), dims, xt, out)
    got = out.cpu().numpy()
    assert np.linalg.norm(got - ref) < 1e-3 * np.linalg.norm(ref)
