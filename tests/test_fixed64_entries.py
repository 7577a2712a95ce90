"""The FP64 stencil entry by entry: the real and the imaginary part of every entry against the oracle, within the
rounding of FP64 sums over that part's own terms.

T = |D| |x| is formed here with the absolute values of the operator's and the vector's real and imaginary parts, as
the real 2 x 2 blocks of a complex product combine them. A part of an entry has at most 80 terms; each is rounded at
2^-53 a few times on its way into the sum. 80 x 2^-53 T on either side (oracle and library) bounds the difference."""
import numpy as np
import pytest

import synth
from oracle import dirac, doublet
from tests.gpu_util import from_dev, to_dev, torch_cuda

L = (6, 2, 4, 10)
KAPPA = 0.126
BOUND = 2 * 80 * 2.0 ** -53


def _mul(spec, M, x):
    """|M| |x| on pairs of absolute real and imaginary parts"""
    r, i = np.abs(M.real), np.abs(M.imag)
    return (np.einsum(spec, r, x[0]) + np.einsum(spec, i, x[1]), np.einsum(spec, r, x[1]) + np.einsum(spec, i, x[0]))


def _terms(op, x, mu):
    """the sums of the absolute terms of the real and imaginary parts of D(mu) x"""
    p = (np.abs(x.real), np.abs(x.imag))
    shp = x.shape
    C = op.C + op.diag * np.eye(12)
    t = [a.reshape(shp) for a in _mul("...ij,...j->...i", C, tuple(a.reshape(shp[:-2] + (12,)) for a in p))]
    m = np.abs(mu).reshape((-1,) + (1,) * (x.ndim - 1))
    t[0], t[1] = t[0] + m * p[1], t[1] + m * p[0]
    for nu in range(4):
        for sign, shift, W in ((-1, dirac.shift_fwd, op.U[..., nu, :, :]), (1, dirac.shift_bwd, op.Ubwd[nu])):
            h = _mul("...ab,...sb->...sa", W, tuple(shift(a, nu, 1) for a in p))
            h = _mul("st,...tc->...sc", op.eye4 + sign * op.g[nu], h)
            t[0], t[1] = t[0] + 0.5 * h[0], t[1] + 0.5 * h[1]
    return t


def _check(y, ref, t):
    for part, T in ((lambda z: z.real, t[0]), (lambda z: z.imag, t[1])):
        assert np.all(np.abs(part(y) - part(ref)) <= BOUND * T)


def _inputs(kind):
    rng = np.random.RandomState(9)
    U = synth.gauge_field(L, 0.25, seed=17)
    x = synth.gaussian_spinors(L, 3, seed=18)
    mu = np.array([0.003, -0.2, 0.0])
    c_sw = 1.0
    if kind == "colours":  # unit links, no clover: each colour is a problem of its own size
        U, c_sw = synth.unit_gauge(L), 0.0
        x = x * 10.0 ** np.array([0.0, -9.0, -18.0])
    elif kind == "parts":  # imaginary parts far below the real ones, links and masses real, few hops mix them
        U, c_sw, mu = synth.unit_gauge(L), 0.0, np.zeros(3)
        x = x.real * 10.0 ** rng.randint(-3, 3, size=x.shape) + 1e-17j * x.imag
    elif kind == "decades":  # every entry of its own size
        x = x * 10.0 ** rng.uniform(-12, 12, size=x.shape)
    elif kind == "sites":
        x = x * 10.0 ** rng.uniform(-12, 12, size=x.shape[:5])[..., None, None]
    elif kind == "sparse":  # one spin, and of one system a single entry
        x[..., 1:, :] = 0.0
        x[1] = 0.0
        x[1, 3, 1, 1, 2, 2, 1] = 1.0 + 1e-30j
    elif kind == "links":  # not unitary, of different sizes, one of them zero
        U = U * 10.0 ** rng.uniform(-3, 3, size=U.shape[:5])[..., None, None]
        U[3, 1, 0, 2, 1] = 0.0
    elif kind == "entries":  # the entries of a link over many decades
        U = U * 10.0 ** rng.uniform(-14, 0, size=U.shape)
    elif kind == "tiny":  # at the lower end of the range of numbers
        x = x * 1e-290
    return U, x, mu, c_sw


KINDS = ["plain", "colours", "parts", "decades", "sites", "sparse", "links", "entries", "tiny"]


def test_the_bound_is_one():
    # at most entries the bound is far below the entry itself: a wrong term would show
    for kind in KINDS:
        U, x, mu, c_sw = _inputs(kind)
        op = dirac.Operator(U, KAPPA, c_sw)
        y, t = op.apply(x, mu), _terms(op, x, mu)
        _check(y, y, t)
        big = t[0] > 0
        assert big.mean() > 0.3 and np.mean(BOUND * t[0][big] <= 1e-9 * np.abs(y.real[big])) > 0.9, kind


def _bundle(T, torch, ctx, x):
    b = torch.empty(T.tmamg_bundle_bytes(ctx, x.shape[0], 64) // 8, dtype=torch.float64, device="cuda")
    T.tmamg_pack(ctx, to_dev(x), b, x.shape[0], 64)
    return b


@pytest.mark.gpu
@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("kind", KINDS)
def test_entries(kind, variant):
    U, x, mu, c_sw = _inputs(kind)
    torch = torch_cuda()
    from paper_2201_03872_gb300 import tmamg as T
    ctx = T.tmamg_create(L, -1)
    try:
        T.tmamg_load_gauge(ctx, U)
        T.tmamg_set_operator(ctx, KAPPA, c_sw)
        T.tmamg_autotune_force(variant)
        op = dirac.Operator(U, KAPPA, c_sw)
        xd = to_dev(x)
        yd = xd.clone()
        T.tmamg_apply(ctx, xd, yd, 3, mu, 64)
        _check(from_dev(yd, x.shape), op.apply(x, mu), _terms(op, x, mu))
        # a doublet whose flavours are of different sizes
        u, v, m, ep = x[0], x[1] * 1e-6, mu[:1] + 0.1, np.array([0.3])
        xb = _bundle(T, torch, ctx, np.stack([u, v]))
        yb = torch.empty_like(xb)
        T.tmamg_dirac_doublet(ctx, xb, yb, 1, m, ep, 64)
        yf = to_dev(x[:2])
        T.tmamg_unpack(ctx, yb, yf, 2, 64)
        y, ref = from_dev(yf, x[:2].shape), doublet.apply(op, u, v, m[0], ep[0])
        for k, (a, b) in enumerate(((u, v), (v, u))):
            t = _terms(op, a[None], m)
            _check(y[k], ref[k], (t[0][0] + ep[0] * np.abs(b.real), t[1][0] + ep[0] * np.abs(b.imag)))
    finally:
        T.tmamg_autotune_force(-1)
        T.tmamg_destroy(ctx)
