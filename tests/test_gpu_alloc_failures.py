"""Calls whose device allocations fail: the library's own switch makes the k-th allocation (and all after it) report
no memory, for every k that a call reaches. Nothing on the GPU is filled or faulted.

A call that finds no memory says so, and the same call afterwards, with memory, is whole: it leaves nothing half
allocated behind that a later call takes for the whole."""
import numpy as np
import pytest

import synth
from oracle import dirac, doublet
from oracle import nn as onn
from tests.gpu_util import Lattice, from_dev, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

L = (8, 4, 4, 8)
KAPPA = 0.125
ALL = 1 << 30
REFUSALS = 3  # of the copies of the operator: in create, load_gauge and set_operator
U = synth.gauge_field(L, 0.3, seed=401)


class Problem:
    """A context with a two-level setup, one right-hand side and two masses; or one without copies of the operator
    and without a setup."""

    def __init__(self, weights=True, copies=True):
        torch_cuda()
        from paper_2201_03872_gb300 import tmamg as T
        self.T = T
        refuse = 0 if copies else REFUSALS
        T.tmamg_debug_fail_alloc(4, refuse)  # create makes four arrays that it needs, then the copies
        self.lat = Lattice(L, to_dev(U), KAPPA, 1.0)
        assert T.tmamg_debug_fail_alloc(0, 0) == refuse
        self.ctx = self.lat.ctx
        self.mu = np.array([0.01, 0.2])
        self.b = synth.gaussian_spinors(L, 1, seed=403)
        if not copies:
            return
        tv = to_dev(synth.gaussian_spinors(L, 4, seed=402).astype(np.complex64))
        T.tmamg_setup_from_vectors(self.ctx, T.setup_params(agg=(2, 2, 2, 2), nv=4, sap_block=(2, 2, 2, 2)), tv)
        if weights:
            T.tmamg_nn_init(self.ctx, 11)

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


def fp64_application(q):
    """D x in FP64 on two systems and on a doublet, against the oracle."""
    T, torch = q.T, q.lat.torch
    x = synth.gaussian_spinors(L, 2, seed=404)
    xb = torch.empty(T.tmamg_bundle_bytes(q.ctx, 2, 64) // 8, dtype=torch.float64, device="cuda")
    yb, yf = torch.empty_like(xb), to_dev(x)
    T.tmamg_pack(q.ctx, to_dev(x), xb, 2, 64)
    op = dirac.Operator(U, KAPPA, 1.0)
    T.tmamg_dirac(q.ctx, xb, yb, 2, q.mu, 64)
    T.tmamg_unpack(q.ctx, yb, yf, 2, 64)
    y, ref = from_dev(yf, x.shape), op.apply(x, q.mu)
    assert np.linalg.norm(y - ref) <= 1e-14 * np.linalg.norm(ref)  # about 80 roundings at 2^-53 on both sides
    T.tmamg_dirac_doublet(q.ctx, xb, yb, 1, q.mu[:1], np.array([0.3]), 64)
    T.tmamg_unpack(q.ctx, yb, yf, 2, 64)
    ref = np.stack(doublet.apply(op, x[0], x[1], q.mu[0], 0.3))
    assert np.linalg.norm(from_dev(yf, x.shape) - ref) <= 1e-14 * np.linalg.norm(ref)
    return y


def _bundles(q, make, n=1):
    x = make(n)
    x.normal_()
    return x, q.lat.torch.zeros_like(x)


def _fine(q, n):
    return q.lat.fine_bundle(synth.gaussian_spinors(L, n, seed=405))


def _apply(q):
    x = to_dev(q.b)
    q.T.tmamg_apply(q.ctx, x, q.lat.torch.zeros_like(x), 1, q.mu[:1], 64)


def _setup(q):
    q.T.tmamg_setup(q.ctx, q.T.setup_params(agg=(2, 2, 2, 2), nv=4, sap_block=(2, 2, 2, 2), setup_iters=1))


CALLS = {
    "load_gauge": lambda q: (q.T.tmamg_load_gauge(q.ctx, U), q.T.tmamg_set_operator(q.ctx, KAPPA, 1.0)),
    "apply": _apply,
    "sap": lambda q: q.T.tmamg_sap(q.ctx, *_bundles(q, lambda n: _fine(q, n)), 1, q.mu[:1], (2, 2, 2, 2), 1, 2),
    "coarse_apply": lambda q: q.T.tmamg_coarse_apply(q.ctx, 1, *_bundles(q, q.lat.coarse_buffer), 1, q.mu[:1], 16),
    "setup": _setup,
    "solve": lambda q: q.solve(host=True),
    "solve64": lambda q: q.solve(host=True, precision=64),
    "learned step": lambda q: q.solve(use_nn=2),
    "block GMRES": lambda q: q.solve(coarse_solver=1),
    "nn_forward": lambda q: q.T.tmamg_nn_forward(q.ctx, *_bundles(q, lambda n: _fine(q, n)), 1),
    "nn_loss_grad": lambda q: q.T.tmamg_nn_loss_grad(q.ctx, _fine(q, 1), _fine(q, 1), 1),
}


@pytest.mark.parametrize("name", list(CALLS))
def test_an_allocation_that_finds_no_memory_gets_what_the_context_can_spare(name):
    for q, error in every_allocation(Problem, CALLS[name], count=1):
        assert error is None, error
        fp64_application(q)  # with or without the copies of the operator


def test_context_without_room_for_the_copies_of_the_operator():
    torch_cuda()
    from paper_2201_03872_gb300 import tmamg as T
    try:
        for k in range(4):
            T.tmamg_debug_fail_alloc(k, ALL)
            with pytest.raises(T.TmamgError) as e:
                T.tmamg_create(L, -1)
            assert e.value.code == -3
    finally:
        T.tmamg_debug_fail_alloc(0, 0)
    q = Problem(copies=False)
    fp64_application(q)
    q.lat.close()


def test_captured_fp64_application_keeps_its_copies_of_the_operator():
    torch = torch_cuda()
    from paper_2201_03872_gb300 import tmamg as T
    st = torch.cuda.Stream()
    mu = np.array([0.01])
    x = synth.gaussian_spinors(L, 1, seed=406)
    with torch.cuda.stream(st):
        ctx = T.tmamg_create(L, -1, st.cuda_stream)
        T.tmamg_load_gauge(ctx, U)
        T.tmamg_set_operator(ctx, KAPPA, 1.0)
        xb = torch.empty(T.tmamg_bundle_bytes(ctx, 1, 64) // 8, dtype=torch.float64, device="cuda")
        yb = torch.empty_like(xb)
        T.tmamg_pack(ctx, to_dev(x), xb, 1, 64)
        T.tmamg_dirac(ctx, xb, yb, 1, mu, 64)  # the launch variants are timed outside the capture
        st.synchronize()
        ref = yb.clone()
        graph = torch.cuda.CUDAGraph()
        graph.capture_begin(capture_error_mode="thread_local")
        T.tmamg_dirac(ctx, xb, yb, 1, mu, 64)
        graph.capture_end()
        T.tmamg_debug_fail_alloc(0, 1)
        try:  # nothing to spare
            with pytest.raises(T.TmamgError) as e:
                T.tmamg_dirac_eo(ctx, xb, yb, 1, mu, 64)
            assert e.value.code == -3 and T.tmamg_debug_fail_alloc(0, 0) == 1
        finally:
            T.tmamg_debug_fail_alloc(0, 0)
        taken = torch.full((1 << 24,), float("nan"), device="cuda")  # memory that a copy given back would be in
        for _ in range(2):
            yb.zero_()
            graph.replay()
            st.synchronize()
            assert torch.equal(yb, ref)
        del taken
        T.tmamg_destroy(ctx)


def test_copies_of_the_operator_are_made_again_after_a_call_that_failed():
    q = Problem()
    T = q.T
    try:
        y = fp64_application(q)
        x = q.lat.torch.zeros(T.tmamg_bundle_bytes(q.ctx, 2, 64) // 8, dtype=q.lat.torch.float64, device="cuda")
        T.tmamg_debug_fail_alloc(0, 2)  # the scratch bundle, with and without the copies
        with pytest.raises(T.TmamgError) as e:
            T.tmamg_dirac_eo(q.ctx, x, q.lat.torch.zeros_like(x), 2, q.mu, 64)
        assert e.value.code == -3 and T.tmamg_debug_fail_alloc(0, 0) == 2
        assert np.array_equal(fp64_application(q), y)
    finally:
        T.tmamg_debug_fail_alloc(0, 0)
        q.lat.close()


@pytest.mark.parametrize("call", ["load_gauge", "set_operator", "setup"])
def test_copies_of_the_operator_are_made_again_with_a_new(call):
    q = Problem()
    y = fp64_application(q)
    q.lat.close()
    q = Problem(copies=False)
    assert not np.array_equal(fp64_application(q), y)  # FP64 arithmetic rounds differently
    if call == "set_operator":
        q.T.tmamg_set_operator(q.ctx, KAPPA, 1.0)
    else:
        CALLS[call](q)
    assert np.array_equal(fp64_application(q), y)
    q.lat.close()
