"""The FP64 stencil's block fixed-point form at the edges of its range, against the FP64 oracle.

The oracle's own sums are FP64, so the tolerance is its rounding: at most 80 terms per entry, each
rounded at 2^-53, relative to the largest term, i.e. 80 x 2^-53 < 1e-14 times (10 + |mu| + eps) times the
largest spinor entry among a site and its neighbours times the largest link row sum."""
import numpy as np
import pytest

import synth
from oracle import dirac, doublet
from tests.gpu_util import from_dev, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

L = (6, 2, 4, 10)  # a direction of two sites (both hops reach the same neighbour), ragged CTAs


def _ctx(U, kappa=0.126, c_sw=1.0):
    torch_cuda()
    from paper_2201_03872_gb300 import tmamg as T
    ctx = T.tmamg_create(L, -1)
    T.tmamg_load_gauge(ctx, U)
    T.tmamg_set_operator(ctx, kappa, c_sw)
    return T, ctx


def _apply(U, x, mu):
    T, ctx = _ctx(U)
    try:
        xd = to_dev(x)
        yd = xd.clone()
        T.tmamg_apply(ctx, xd, yd, x.shape[0], mu, 64)
        return from_dev(yd, x.shape)
    finally:
        T.tmamg_destroy(ctx)


def _near(x):
    """largest entry (absolute) among a site and its neighbours, [n, T, Z, Y, X]"""
    m = np.maximum(np.abs(x.real), np.abs(x.imag)).max(axis=(-1, -2))
    out = m
    for ax in range(1, 5):
        out = np.maximum(out, np.maximum(np.roll(m, 1, ax), np.roll(m, -1, ax)))
    return out


def _inputs(kind):
    rng = np.random.RandomState(5)
    U = synth.gauge_field(L, 0.25, seed=7)
    x = synth.gaussian_spinors(L, 3, seed=8)
    mu = np.array([0.003, -0.2, 0.05])
    if kind == "wide":  # magnitudes over 24 decades from site to site
        x = x * 10.0 ** rng.uniform(-12, 12, size=x.shape[:5])[..., None, None]
    elif kind == "point":  # zero sites, components and signs of zero
        y = np.zeros_like(x)
        y[:, 0, 0, 0, 0, 1, 2] = 1.0
        y[:, 5, 3, 1, 2, 3, 0] = -0.0
        x = y
    elif kind == "huge":  # beyond the fixed-point range: FP64 arithmetic
        x = x * 1e290
    elif kind == "tiny":
        x = x * 1e-290
    elif kind == "mass":  # |mu| as large as the clover block on some systems
        mu = np.array([50.0, 0.01, -3.0])
    elif kind == "links":  # not unitary, of different sizes, one of them zero
        U = U * 10.0 ** rng.uniform(-3, 3, size=U.shape[:5])[..., None, None]
        U[3, 1, 0, 2, 1] = 0.0
    return U, x, mu


@pytest.mark.parametrize("kind", ["plain", "wide", "point", "huge", "tiny", "mass", "links"])
def test_fixed_point_stencil_edges(kind):
    U, x, mu = _inputs(kind)
    y = _apply(U, x, mu)
    ref = dirac.Operator(U, 0.126, 1.0).apply(x, mu)
    scale = max(1.0, np.abs(U).max() * 3) ** (4 if kind == "links" else 1)  # the clover holds products of four links
    bound = 1e-14 * (10.0 + np.abs(mu).max()) * scale * _near(x)[..., None, None]
    assert np.all(np.abs(y - ref) <= bound + 1e-300)
    if kind == "point":
        far = _near(x) == 0.0
        assert far.any() and np.all(y[far] == 0.0)


def test_non_finite_entries_stay_with_their_system_and_neighbours():
    U, x, mu = _inputs("plain")
    x[1, 2, 1, 0, 3, 2, 1] = np.nan
    x[2, 7, 0, 1, 1, 0, 0] = np.inf
    y = _apply(U, x, mu)
    bad = ~np.isfinite(_near(np.where(np.isfinite(x), 0.0, np.nan)))
    assert np.isfinite(y[~bad]).all() and not np.isfinite(y[bad]).all(axis=(-1, -2)).any()
    ref = dirac.Operator(U, 0.126, 1.0).apply(np.where(np.isfinite(x), x, 0.0), mu)
    assert np.allclose(y[~bad], ref[~bad], rtol=0, atol=1e-12)


def test_doublet_coupling_with_a_partner_of_another_size():
    # the partner's entries need a larger exponent than the site's own stencil, and the other way round
    U, x, _ = _inputs("plain")
    torch = torch_cuda()
    T, ctx = _ctx(U)
    try:
        xs = np.concatenate([x[:1], x[1:2] * 1e9, x[2:3] * 1e9, x[:1]])
        mu, eps = np.array([0.02, 0.1]), np.array([0.3, 0.07])
        nb = T.tmamg_bundle_bytes(ctx, 4, 64) // 8
        xb = torch.empty(nb, dtype=torch.float64, device="cuda")
        yb = torch.empty_like(xb)
        yd = to_dev(xs)
        T.tmamg_pack(ctx, to_dev(xs), xb, 4, 64)
        T.tmamg_dirac_doublet(ctx, xb, yb, 2, mu, eps, 64)
        T.tmamg_unpack(ctx, yb, yd, 4, 64)
        y = from_dev(yd, xs.shape)
        op = dirac.Operator(U, 0.126, 1.0)
        near = _near(xs)
        for q in range(2):
            u, d = doublet.apply(op, xs[2 * q], xs[2 * q + 1], mu[q], eps[q])
            for f, ref in ((0, u), (1, d)):
                top = np.maximum(near[2 * q + f], eps[q] * near[2 * q + 1 - f])
                assert np.all(np.abs(y[2 * q + f] - ref) <= 1e-13 * 11.0 * top[..., None, None])
    finally:
        T.tmamg_destroy(ctx)
