"""Calls whose device allocations fail: the library's own switch makes the k-th allocation (and all after it) report
no memory, for every k that a call reaches. Nothing on the GPU is filled or faulted.

A call that finds no memory says so, and the same call afterwards, with memory, is whole: it leaves nothing half
allocated behind that a later call takes for the whole."""
import numpy as np
import pytest

import synth
from oracle import dirac
from oracle import nn as onn
from tests.gpu_util import Lattice, from_dev, to_dev

pytestmark = pytest.mark.gpu

L = (8, 4, 4, 8)
KAPPA = 0.125
ALL = 1 << 30
U = synth.gauge_field(L, 0.3, seed=401)


class Problem:
    """A context with a two-level setup, one right-hand side and two masses."""

    def __init__(self, agg=(2, 2, 2, 2), weights=True):
        self.lat = Lattice(L, U, KAPPA, 1.0)
        T = self.T = self.lat.T
        self.ctx = self.lat.ctx
        tv = to_dev(synth.gaussian_spinors(L, 4, seed=402).astype(np.complex64))
        T.tmamg_setup_from_vectors(self.ctx, T.setup_params(agg=agg, nv=4, sap_block=(2, 2, 2, 2)), tv)
        if weights:
            T.tmamg_nn_init(self.ctx, 11)
        self.mu = np.array([0.01, 0.2])
        self.b = synth.gaussian_spinors(L, 1, seed=403)

    def solve(self, host=False, **kw):
        p = self.T.solve_params(tol=1e-10, **kw)
        if host:
            b, x = np.ascontiguousarray(self.b), np.zeros((2,) + self.b.shape[1:], dtype=np.complex128)
            self.T.tmamg_solve(self.ctx, b, 1, self.mu, 2, x, 0, p)
        else:
            b = to_dev(self.b)
            x = self.lat.torch.zeros(2 * b.numel(), dtype=b.dtype, device="cuda")
            self.T.tmamg_solve(self.ctx, b, 1, self.mu, 2, x, 1, p)
            x = from_dev(x, (2,) + self.b.shape[1:])
        op = dirac.Operator(U, KAPPA, 1.0)
        res = [np.linalg.norm(op.apply(x[k:k + 1], self.mu[k:k + 1]) - self.b) for k in range(2)]
        assert max(res) <= 2e-10 * np.linalg.norm(self.b), res  # the solver's goal, and the oracle's rounding


def every_allocation(make, call, count=ALL):
    """call(problem) with its k-th allocation and the count - 1 after it failing, for k = 0, 1, ... (every third from
    9 on) until it reaches none: yields (problem, error or None) while the switch is off again."""
    for k in list(range(9)) + list(range(9, 1000, 3)):
        q = make()
        try:
            error = None
            q.T.tmamg_debug_fail_alloc(k, count)
            try:
                call(q)
            except q.T.TmamgError as e:
                error = e
            failed = q.T.tmamg_debug_fail_alloc(0, 0)
            if not failed:
                assert error is None and k > 0
                return
            yield q, error
        finally:
            q.T.tmamg_debug_fail_alloc(0, 0)
            q.lat.close()
    raise AssertionError("the call never ran out of allocations")


@pytest.mark.parametrize("kw", [dict(use_nn=2), dict(coarse_solver=1), dict(coarse_solver=2), dict(precision=64),
                                dict(precision=64, host=True)],
                         ids=["learned step", "block GMRES", "GMRES per step", "FP64", "FP64 host"])
def test_solve_after_a_solve_without_memory(kw):
    for q, error in every_allocation(Problem, lambda q: q.solve(**kw)):
        assert error is not None and error.code == -3, error
        q.solve(**kw)


def test_network_weights_after_a_failure():
    W = onn.init_weights(seed=11, scale=1.0, identity=True)
    for q, error in every_allocation(lambda: Problem(weights=False), lambda q: q.T.tmamg_nn_set_weights(q.ctx, W)):
        assert error is not None and error.code == -3, error
        q.T.tmamg_nn_set_weights(q.ctx, W)
        assert np.allclose(q.T.tmamg_nn_get_weights(q.ctx), np.concatenate([np.ravel(w) for w in W]), atol=1e-6)
        r = q.lat.fine_bundle(q.b)
        y = q.lat.torch.zeros_like(r)
        q.T.tmamg_nn_forward(q.ctx, r, y, 1, bf16=True)
        assert np.isfinite(q.lat.from_fine_bundle(y, 1)).all()
