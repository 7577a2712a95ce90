"""SAP on block shapes at the edges of the kernels' paths, against the FP64 oracle: extents of one (a site
crosses a face both ways), of two, blocks that span the lattice in some or all directions, block volumes
that are no multiple of a warp, a ragged last tile; one cycle (every correction is fresh) and several.
Tolerance as in the other SAP tests: FP32 rounding through a few MR steps, 2e-5."""
import numpy as np
import pytest

import synth
from oracle import dirac, sap
from tests.gpu_util import Lattice, relerr

pytestmark = pytest.mark.gpu
TOL32 = 2e-5


M = (8, 4, 4, 8)


@pytest.mark.parametrize("L,block,cycles,steps,nsys", [
    (M, (1, 4, 4, 2), 2, 3, 3), (M, (2, 1, 2, 1), 1, 2, 2), (M, (2, 2, 2, 2), 3, 4, 5), (M, (8, 2, 4, 4), 2, 5, 1),
    (M, (4, 4, 2, 8), 1, 1, 4), (M, (8, 4, 4, 2), 2, 4, 7), ((12, 4, 4, 8), (3, 2, 2, 1), 2, 3, 2),
    ((4, 4, 2, 8), (4, 4, 2, 8), 2, 3, 3),
])
def test_sap_block_shapes(L, block, cycles, steps, nsys):
    U = synth.gauge_field(L, 0.3, seed=61)
    kappa, c_sw = 0.126, 1.0
    lat = Lattice(L, U, kappa, c_sw)
    try:
        r = synth.gaussian_spinors(L, nsys, seed=62).astype(np.complex64).astype(np.complex128)
        mu = np.linspace(0.002, 0.2, nsys)
        rb = lat.fine_bundle(r)
        eb = lat.torch.full_like(rb, 3.0)  # whatever e held before is no part of the result
        lat.T.tmamg_sap(lat.ctx, rb, eb, nsys, mu, block, cycles, steps)
        e = lat.from_fine_bundle(eb, nsys)
        op = dirac.Operator(U, kappa, c_sw)
        want = sap.sap(op, r, mu, block, cycles, steps)
        for n in range(nsys):
            assert relerr(e[n], want[n]) <= TOL32, n
    finally:
        lat.close()
