"""The persistent coarse solver at the edges of its vector phases: residuals of converged solves.

256 sites of 2 nv = 2 to 64 unknowns: tiles below, at and above the entries that a block's threads own at once, one
system (a tile over all blocks), twelve, and seventy (more than a pass of four lanes per system holds); cycles
shorter and longer than the basis vectors that shared memory caches between the two passes, with restarts.

FP32: the solver's goal 1e-5 within a factor of two for the FP32 operator's own rounding. FP16: the goal 1e-2 holds for
the rounded operator; its difference on x is measured, and every one of the `it` basis vectors adds one like it."""
import numpy as np
import pytest

import synth
from tests.gpu_util import Lattice, coarse_from_bundle, coarse_to_bundle, torch_cuda

pytestmark = pytest.mark.gpu
L = (8, 8, 8, 8)


@pytest.mark.parametrize("nv,nsys,restart", [(1, 1, 5), (8, 12, 40), (8, 70, 40), (9, 70, 3), (24, 12, 40), (32, 2, 30), (32, 70, 16)])
def test_converged_residuals(nv, nsys, restart):
    torch = torch_cuda()
    lat = Lattice(L, synth.gauge_field(L, 0.3, seed=3), 0.125, 1.0)
    try:
        T = lat.T
        tv = synth.gaussian_spinors(L, nv, seed=5).astype(np.complex64)
        p = T.setup_params(nv=nv, agg=(2, 2, 2, 2), sap_block=(2, 2, 2, 2))
        T.tmamg_setup_from_vectors(lat.ctx, p, torch.from_numpy(tv.view(np.float32).copy()).cuda())
        Vc, nc = int(np.prod(L)) // 16, 2 * nv
        rc = synth.complex_normal(105, 1, (nsys, Vc, nc)).astype(np.complex64)
        rc[-1] *= 1e-4
        mu = np.array([0.02])
        rb = torch.from_numpy(coarse_to_bundle(rc, nc, Vc)).cuda()

        def field(b):
            torch.cuda.synchronize()
            return coarse_from_bundle(b.cpu().numpy(), nsys, nc, Vc).reshape(nsys, -1)

        for prec, tol in ((32, 1e-5), (16, 1e-2)):
            xb, yb, zb = (torch.zeros_like(rb) for _ in range(3))
            sp = T.solve_params(coarse_solver=0, coarse_tol=tol, coarse_restart=restart, coarse_maxiter=400, coarse_precision=prec)
            it = T.tmamg_coarse_solve(lat.ctx, 1, rb, xb, nsys, mu, 1, sp)
            T.tmamg_coarse_apply(lat.ctx, 1, xb, yb, nsys, np.full(nsys, mu[0]), 32)
            T.tmamg_coarse_apply(lat.ctx, 1, xb, zb, nsys, np.full(nsys, mu[0]), 16)
            y, z = field(yb), field(zb)
            for n in range(nsys):
                b = rc[n].astype(complex).ravel()
                res, pert = (np.linalg.norm(v) / np.linalg.norm(b) for v in (b - y[n], z[n] - y[n]))
                assert res <= (2 * tol if prec == 32 else 1.05 * tol + (1 + np.sqrt(it)) * pert), (prec, n, it, res, pert)
    finally:
        lat.close()
