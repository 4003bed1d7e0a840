"""GPU tests of the FP64 operators on fields whose components differ widely in
size within one 5D site: the real and the imaginary part of every output
component keep FP64 precision relative to the terms that make them up, however
large the other components are.

Bound.  Let |K| be the operator on (real, imaginary) pairs with every matrix
element (of M, D~, the links and the spin projectors) replaced by its absolute
value.  FP64 arithmetic gives |error| <= n 2^-53 |K||x| with n below 64 (the
longest chain of rounded operations of one output).  The fixed-point sums of
the hop are off by at most 96 units a real (per direction: 4.9 from the inputs,
1.2 from the alignment, 2.8 from the low products, 3 from the links) and are
only taken where one of the real's eight terms U h is at least 2^51 units, so
by at most 96 2^-51 = 384 2^-53 of the sum of the terms' sizes; D~^T in K^dag
passes that on as it is.  Both together stay below 512 2^-53 |K||x|, and a real
that is made of zeros is zero.
"""
import numpy as np
import pytest

from paper_1706_05843_gb300 import inputs as I

pytestmark = pytest.mark.gpu

ACT = dict(M5=1.8, b=1.5, c=0.5, m1=0.04, m2=1.0, m3=0.04, beta=-1.0, pm=1, t_bc=-1)
BOUND = 512 * 2.0 ** -53


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


def links(dims, kind):
    """SU(3) links: generic, diagonal, diagonal up to 1e-9 (a weak field), or diagonal with elements 1 and -1."""
    if kind == "generic":
        return I.gauge_field(dims, 0.5, 3)
    rng = np.random.default_rng(4)
    shape = tuple(dims[::-1]) + (4,)
    ph = rng.uniform(-np.pi, np.pi, shape + (2,))
    d = np.exp(1j * np.concatenate([ph, -ph.sum(-1, keepdims=True)], -1))
    if kind == "signs":
        d = np.sign(d.real) + 0j
    e = 1e-9 if kind == "weak" else 0.0
    # rows 0 and 1 orthonormal to 1e-18, row 2 their conjugate cross product
    off = e * (rng.standard_normal(shape + (3, 2)) @ [1, 1j])
    r0 = np.stack([d[..., 0], off[..., 0], off[..., 1]], -1)
    r1 = np.stack([-off[..., 0].conj() * d[..., 0] * d[..., 1], d[..., 1], off[..., 2]], -1)
    return np.stack([r0, r1, np.cross(r0, r1).conj()], -2)


def fields(dims, Ls, kind):
    x = I.gaussian_fermion(dims, Ls, 1001)
    if kind == "colour":
        x *= np.array([1.0, 1e-6, 1e-12])
    elif kind == "colour18":
        x *= np.array([1e-18, 1.0, 1e-9])
    elif kind == "one colour":
        x[..., 1:] = 0.0
    elif kind == "point":
        keep = x[1, 0, 1, 0, 1, 2, 1]
        x = np.zeros_like(x)
        x[1, 0, 1, 0, 1, 2, 1] = keep.real
    elif kind == "spin":
        x *= np.array([1.0, 1e-10, 1e-10, 1e-10])[:, None]
    elif kind == "spin pair":
        x *= np.array([1e-7, 1.0, 1e-7, 1e-7])[:, None]
    elif kind == "real":
        x *= np.array([1.0, 1.0, 1e-9, 1e-9])[:, None]
        x.imag *= 1e-9
    return x


def smatrices(act, Ls):
    """(M, D~, D~^-1) in s, each for chirality + and -."""
    b, c, M5, m1, m2, m3, pm = (act[k] for k in ("b", "c", "M5", "m1", "m2", "m3", "pm"))
    L = np.eye(Ls, k=-1)
    L[0, -1] = -m1
    N = lambda m: b ** Ls + m * c ** Ls
    k = (b + c) * (m3 - m2) * b ** (2 * Ls) / (N(m2) * N(m3))
    s = np.arange(Ls)
    shift = np.zeros((2, Ls, Ls))
    if pm > 0:
        shift[0][:, -1] = (-c) ** s / b ** (Ls + s + 1) * N(m1) * k
    else:
        shift[1][:, 0] = -(-1.0) ** s * c ** (Ls - 1 - s) / b ** (2 * Ls - s) * N(m1) * k
    E = np.eye(Ls)
    M = [(b * (4 - M5) + 1) * E + (c * (4 - M5) - 1) * A + pm * act["beta"] * S for A, S in zip((L, L.T), shift)]
    D = [b * E + c * A for A in (L, L.T)]
    return M, D, [np.linalg.inv(d) for d in D]


def in_s(mats, x, adjoint=False):
    m = np.abs(np.stack(mats))
    if adjoint:
        m = m.transpose(0, 2, 1)
    return np.concatenate([np.einsum("st,...tacr->...sacr", m[0], x[..., :2, :, :]),
                           np.einsum("st,...tacr->...sacr", m[1], x[..., 2:, :, :])], -3)


def hop(U, x, gmask=0):
    """sum_mu (1 + |gamma_mu|) (|U_mu(x)| x(x + mu) + |U_mu(x - mu)|^T x(x - mu)), x (F, T, Z, Y, X, s, 4, 3, 2)."""
    A, out = (np.abs(U.real), np.abs(U.imag)), np.zeros_like(x)

    def link(mu, sub, v):
        eq = f"tzyx{sub},ftzyxspbr->ftzyxspar"
        return np.einsum(eq, A[0][..., mu, :, :], v) + np.einsum(eq, A[1][..., mu, :, :], v[..., ::-1])

    for mu in range(4):
        ax = 4 - mu
        f, b = np.roll(x, -1, ax), np.roll(link(mu, "ba", x), 1, ax)
        if (gmask >> mu) & 1:  # the other flavour across the boundary
            at = lambda i: (slice(None),) * ax + (i,)
            f[at(-1)] = f[at(-1)][::-1].copy()
            b[at(0)] = b[at(0)][::-1].copy()
        w = link(mu, "ab", f) + b
        g = w[..., [3, 2, 1, 0] if mu < 2 else [2, 3, 0, 1], :, :]
        out += w + (g[..., ::-1] if mu in (0, 2) else g)
    return out


def pairs(x):
    return np.stack([x.real, x.imag], -1)


def majorant(which, act, U, x, gmask=0):
    Ls = x.shape[-3]
    M, D, Di = smatrices(act, Ls)
    a = np.abs(pairs(x if gmask else x[None]))
    if which == "kdag":
        r = in_s(M, a, True) + 0.5 * in_s(D, hop(U, a, gmask), True)
    else:
        if which == "h":
            a = in_s(Di, a)
        r = in_s(M, a) + 0.5 * hop(U, in_s(D, a), gmask)
        if which == "h":
            r = r[..., ::-1, :, :, :]
    return r if gmask else r[0]


def worst(got, ref, maj):
    d = np.abs(pairs(got - ref))
    assert np.all(d[maj == 0.0] == 0.0)
    return np.max(d / np.where(maj == 0.0, 1.0, maj))


CASES = [
    ((4, 2, 4, 6), 4, 1, "diagonal", "colour"),
    ((4, 4, 2, 4), 8, -1, "diagonal", "colour18"),
    ((2, 4, 4, 2), 12, 1, "weak", "colour"),
    ((4, 4, 4, 4), 8, 1, "weak", "one colour"),
    ((4, 4, 2, 2), 12, -1, "generic", "spin"),
    ((2, 2, 4, 4), 16, 1, "generic", "spin pair"),
    ((2, 4, 2, 4), 8, 1, "signs", "real"),
    ((4, 2, 4, 4), 8, 1, "signs", "one colour"),
    ((4, 4, 4, 2), 12, -1, "signs", "point"),
    ((4, 4, 4, 4), 4, 1, "weak", "point"),
    ((6, 2, 4, 4), 4, -1, "generic", "plain"),
]


@pytest.mark.parametrize("dims,Ls,pm,link,field", CASES)
@pytest.mark.parametrize("which", ["k", "kdag", "h"])
@pytest.mark.parametrize("overlap", [False, True])
def test_components_keep_fp64_precision(env, dims, Ls, pm, link, field, which, overlap):
    torch, B, O = env
    act = dict(ACT, pm=pm)
    U, x = links(dims, link), fields(dims, Ls, field)
    o = O.Oracle(O.Action(dims=dims, Ls=Ls, **act), U)
    ref = {"k": o.k, "kdag": lambda v: o.k(v, dag=True), "h": o.hsys}[which](x)
    s = B.Solver(U, dims, Ls, **act)
    buf = torch.empty(x.size + 12, dtype=torch.complex128, device="cuda")
    xin = buf[:x.size].view(x.shape)
    xin.copy_(torch.from_numpy(x))
    out = buf[12:].view(x.shape) if overlap else torch.empty_like(xin)
    {"k": B.eofa_apply, "kdag": B.eofa_apply_dag, "h": B.eofa_apply_h}[which](s.ctx, xin, out)
    got = out.cpu().numpy()
    s.close()
    e = worst(got, ref, majorant(which, act, U, x))
    print(f"{which} {dims} {Ls} {link} {field}: {e:.2e}")
    assert e <= BOUND


@pytest.mark.parametrize("dims,Ls,pm,link,field", CASES[:4])
def test_noalloc_components(env, dims, Ls, pm, link, field):
    torch, B, O = env
    act = dict(ACT, pm=pm)
    U, x = links(dims, link), fields(dims, Ls, field)
    xt = torch.from_numpy(x).cuda()
    out = torch.empty_like(xt)
    B.eofa_apply_noalloc(B.make_params(dims, Ls, **act), torch.from_numpy(U).cuda(), xt, out)
    got = out.cpu().numpy()
    ref = O.Oracle(O.Action(dims=dims, Ls=Ls, **act), U).k(x)
    assert worst(got, ref, majorant("k", act, U, x)) <= BOUND


@pytest.mark.parametrize("gmask", [7, 8])
def test_gparity_components(env, gmask):
    torch, B, O = env
    from oracle.gparity import GOracle
    dims, Ls = (4, 2, 4, 4), 8
    U = links(dims, "weak")
    x = np.stack([fields(dims, Ls, "colour"), fields(dims, Ls, "one colour")])
    s = B.Solver(U, dims, Ls, gparity=gmask, **ACT)
    got = s.apply_h(torch.from_numpy(x).cuda()).cpu().numpy().reshape(x.shape)
    s.close()
    ref = GOracle(O.Action(dims=dims, Ls=Ls, **ACT), U, gmask).hsys(x)
    assert worst(got, ref, majorant("h", ACT, U, x, gmask)) <= BOUND


@pytest.mark.parametrize("dims,Ls,pm,link,field", CASES)
def test_fp64_solve(env, dims, Ls, pm, link, field):
    """The kernels of the FP64 CG, whose hops hand their output on as integers
    and doubles, on the same fields: a solve to 1e-12 judged by the oracle."""
    torch, B, O = env
    act = dict(ACT, pm=pm, m1=0.2, m3=0.2)
    U, x = links(dims, link), fields(dims, Ls, field)
    s = B.Solver(U, dims, Ls, **act)
    sol, st = s.solve(torch.from_numpy(x).cuda(), tol=1e-12, inner="f64")
    sol = sol.cpu().numpy()
    s.close()
    r = x - O.Oracle(O.Action(dims=dims, Ls=Ls, **act), U).hsys(sol)
    print(f"{dims} {Ls} {link} {field}: {st.inner_iters} iterations")
    assert np.linalg.norm(r) <= 1e-12 * np.linalg.norm(x)
