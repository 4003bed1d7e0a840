"""GPU tests of the FP64 hop's fixed-point arithmetic at the edges of its range.

The kernels keep a hop input as 57-bit integers under one exponent per 5D
site and take sites with Inf, NaN or extreme magnitudes through FP64
arithmetic; the oracle's plain FP64 operator is the reference.

Bound of the elementwise comparison: an output of K is a sum of a few hundred
products whose coefficients add up to less than 64 in size (b (4 - M5) + 1,
the eight hops with b + c, the shift), each product and each rounding off by
at most 2^-53 of the largest input in reach, S: |difference| <= 64 * 16 *
2^-53 S = 1.2e-13 S covers both sides.
"""
import numpy as np
import pytest

from paper_1706_05843_gb300 import inputs as I

pytestmark = pytest.mark.gpu

ACT = dict(M5=1.8, b=1.5, c=0.5, m1=0.04, m2=1.0, m3=0.04, beta=-1.0, pm=1, t_bc=-1)
BOUND = 64 * 16 * 2.0 ** -53


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1706_05843_gb300 import build
    build.build()
    from paper_1706_05843_gb300 import binding as B
    import oracle
    oracle.build()
    return torch, B, oracle


def reach(x):
    """Largest |x| over all slices and components of each 4D site and its eight neighbours."""
    a = np.abs(x).max(axis=(4, 5, 6))
    out = a.copy()
    for ax in range(4):
        for d in (1, -1):
            out = np.maximum(out, np.roll(a, d, ax))
    return out


@pytest.mark.parametrize("dims,Ls,lo,hi", [
    ((4, 4, 4, 4), 4, 0, 0),          # plain
    ((4, 2, 6, 4), 8, -9, 9),         # exponents that differ from site to site within the 57 bits
    ((4, 4, 2, 4), 12, -40, 40),      # neighbours shifted out altogether
    ((2, 4, 4, 2), 16, -330, 290),    # subnormals and magnitudes on the FP64 path beside fixed point
])
@pytest.mark.parametrize("dag", [False, True])
def test_magnitudes(env, dims, Ls, lo, hi, dag):
    torch, B, O = env
    U = I.gauge_field(dims, 0.5, 3)
    x = I.gaussian_fermion(dims, Ls, 1001)
    rng = np.random.default_rng(5)
    x = x * 10.0 ** rng.integers(lo, hi + 1, size=x.shape[:5] + (1, 1))
    if lo == 0:
        x[:, :, :, 0] = 0.0  # zero neighbours
    o = O.Oracle(O.Action(dims=dims, Ls=Ls, **ACT), U)
    ref = o.k(x, dag=dag)
    s = B.Solver(U, dims, Ls, **ACT)
    got = s.apply(torch.from_numpy(x).cuda(), dag=dag).cpu().numpy()
    s.close()
    S = reach(x)[..., None, None, None]
    tiny = 64 * 16 * 64 * 5e-324  # the same count of subnormal roundings, each scaled by at most 64
    assert np.all(np.abs(got - ref) <= BOUND * S + tiny)


def test_powers_of_two_are_exact(env):
    torch, B, O = env
    dims, Ls = (4, 4, 4, 4), 8
    s = B.Solver(I.gauge_field(dims, 0.5, 3), dims, Ls, **ACT)
    x = torch.from_numpy(I.gaussian_fermion(dims, Ls, 1001)).cuda()
    ref = s.apply(x)
    for k in (-900, -30, 1, 64, 900):
        assert torch.equal(s.apply(x * 2.0 ** k), ref * 2.0 ** k)
    s.close()


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_non_finite_stays_local(env, bad):
    torch, B, O = env
    dims, Ls = (4, 4, 4, 4), 4
    s = B.Solver(I.gauge_field(dims, 0.5, 3), dims, Ls, **ACT)
    x = I.gaussian_fermion(dims, Ls, 1001)
    ref = s.apply(torch.from_numpy(x).cuda()).cpu().numpy()
    site, sl = (1, 2, 3, 0), 2
    x[site + (sl, 1, 2)] = bad
    got = s.apply(torch.from_numpy(x).cuda()).cpu().numpy()
    s.close()
    hit = np.zeros(x.shape[:4], dtype=bool)
    hit[site] = True
    near = hit.copy()
    for ax in range(4):
        for d in (1, -1):
            near |= np.roll(hit, d, ax)
    assert np.array_equal(got[~near], ref[~near])
    assert not np.isfinite(got[near][:, sl]).all(axis=(1, 2)).any()


@pytest.mark.parametrize("which", ["k", "kdag", "h"])
@pytest.mark.parametrize("shift", [0, 24])
def test_canonical_fields(env, which, shift):
    """The applications read and write the caller's fields in place: a ragged
    lattice with Ls = 12 and 16 against the oracle, into a separate field and
    into one that overlaps the input (shift complex elements further on)."""
    torch, B, O = env
    for dims, Ls, pm in (((2, 4, 6, 2), 12, -1), ((6, 2, 2, 4), 16, 1)):
        act = dict(ACT, pm=pm)
        U = I.gauge_field(dims, 0.5, 3)
        x = I.gaussian_fermion(dims, Ls, 1001)
        o = O.Oracle(O.Action(dims=dims, Ls=Ls, **act), U)
        ref = {"k": o.k, "kdag": lambda v: o.k(v, dag=True), "h": o.hsys}[which](x)
        s = B.Solver(U, dims, Ls, **act)
        buf = torch.zeros(x.size + max(shift, 1) * 12, dtype=torch.complex128, device="cuda")
        xin = buf[:x.size].view(x.shape)
        xin.copy_(torch.from_numpy(x))
        out = buf[shift * 12:shift * 12 + x.size].view(x.shape) if shift else torch.empty_like(xin)
        {"k": B.eofa_apply, "kdag": B.eofa_apply_dag, "h": B.eofa_apply_h}[which](s.ctx, xin, out)
        got = out.cpu().numpy()
        s.close()
        assert np.linalg.norm(got - ref) <= 1e-14 * np.linalg.norm(ref)


@pytest.mark.parametrize("dims,Ls", [((4, 4, 4, 4), 4), ((16, 16, 16, 16), 16)])
@pytest.mark.parametrize("shift", [0, 24])
def test_applications_are_capturable(env, dims, Ls, shift):
    """A new context's first application may be a captured one, with both
    parities in one grid and in two, into a separate field and into one that
    overlaps the input; the replay gives the eager result to the last bit."""
    torch, B, _ = env
    s = B.Solver(I.gauge_field(dims, 0.3, 5), dims, Ls, **ACT)
    x = torch.from_numpy(I.gaussian_fermion(dims, Ls, 6)).cuda()
    for f in (B.eofa_apply, B.eofa_apply_dag, B.eofa_apply_h):
        buf = torch.empty(x.numel() + max(shift, 1) * 12, dtype=x.dtype, device="cuda")
        a = buf[:x.numel()].view(x.shape)
        a.copy_(x)
        out = buf[shift * 12:shift * 12 + x.numel()].view(x.shape) if shift else torch.empty_like(a)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            f(s.ctx, a, out)
        g.replay()
        torch.cuda.synchronize()
        ref = torch.empty_like(x)
        f(s.ctx, x, ref)
        assert torch.equal(torch.view_as_real(out), torch.view_as_real(ref))
    s.close()
