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


@pytest.mark.parametrize("dims,S", [
    ((1, 1, 1, 1), 1), ((5, 4, 3, 7), 2), ((66, 2, 2, 2), 1), ((4, 6, 2, 9), 5), ((2, 2, 2, 2), 1),
])
@pytest.mark.parametrize("offset", [0, 1])
def test_net_backward_storage_model(dims, S, offset):
    """Gradients against the FP64 oracle within twice the storage model's own
    distance (test_gpu_learned says why); offset: fields that start on a
    4-byte boundary only."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1706_05843_gb300 import binding as B
    from paper_1706_05843_gb300 import build
    from test_gpu_learned import backward_bf16_storage
    build.build()
    X, Y, Z, T = dims
    rng = np.random.default_rng(8)
    w = N.bf16_round(np.concatenate([rng.standard_normal(81 * co * ci) * np.sqrt(2.0 / (81 * ci))
                                     for ci, co in zip(N.CIN, N.COUT)]))
    x, d = (N.bf16_round(rng.standard_normal((S, T, Z, Y, X, 24))) for _ in range(2))
    dw_ref, dx_ref = N.backward(x, w, d)
    dw_sm, dx_sm = backward_bf16_storage(x, w, d)

    def field(a):
        buf = torch.full((a.size + 4,), float("nan"), device="cuda")
        v = buf[offset:offset + a.size].view(a.shape)
        v.copy_(torch.from_numpy(a.astype(np.float32)))
        return v

    din = field(np.zeros_like(x))
    dw = B.eofa_net_backward(w.astype(np.float32), dims, field(x), field(d), din)
    # where the storage model happens to have no flipped sign, its FP32 sums are off by 1e-6 and its stored
    # BF16 gradients by half a unit, 2^-9
    for got, sm, ref in ((dw, dw_sm, dw_ref), (din.cpu().numpy(), dx_sm, dx_ref)):
        n = np.linalg.norm(ref)
        assert np.linalg.norm(got - ref) <= max(2 * np.linalg.norm(sm - ref), 2.0 ** -9 * n)
