"""Batched norms at the edges of their loops, through the residuals that a solve reports.

768 sites x 12 entries: with one system every thread of the reduction has one entry, with 20 and 40 systems the blocks
per system are fewer and a thread has the first one to three of its four entries in flight. The FP64 norms are
compared with the residual of the returned solution (operator in FP64 on the host): its rounding and the GPU's are
below 1e-13 of |b|. The FP32 norms scale the Krylov vectors, without which the solve would not converge."""
import numpy as np
import pytest

import synth
from oracle import dirac
from tests.gpu_util import Lattice, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [1, 20, 40])
def test_reported_residuals(nrhs):
    torch_cuda()
    L = (12, 4, 4, 4)
    U = synth.gauge_field(L, 0.3, seed=3)
    lat = Lattice(L, U, 0.125, 1.0)
    try:
        T = lat.T
        T.tmamg_setup(lat.ctx, T.setup_params(agg=(2, 2, 2, 2), nv=8, sap_block=(2, 2, 2, 2), setup_iters=2))
        b = synth.gaussian_spinors(L, nrhs, seed=4)
        x = np.zeros((nrhs, 1) + b.shape[1:], dtype=np.complex128)
        rc, stats = T.tmamg_solve(lat.ctx, b, nrhs, [0.02], 1, x, 0, T.solve_params(restart=8, tol=1e-3))
        op = dirac.Operator(U, 0.125, 1.0)
        for n in range(nrhs):
            res = np.linalg.norm(b[n] - op.apply(x[n, 0], 0.02)) / np.linalg.norm(b[n])
            assert res <= 1e-3 and abs(stats[n].true_rel_res - res) <= 1e-13, (n, res, stats[n].true_rel_res)
    finally:
        lat.close()
