"""FP16 coarse operator at the edges of its pipeline, against the FP32 operator on the same level.

Blocks of one to eight row groups (the shared-memory ring holds 16 stages to 3), system counts around the chunks
of 8 and 16, and 16 and 256 sites: fewer than CTAs, and CTAs of one site beside CTAs of two. Both operands are
rounded to FP16, a relative error of at most 2^-10 per product, and 2e-5 is the FP32 operator's: 2e-3 in norm, the
bound that the FP16 operator keeps to elsewhere."""
import numpy as np
import pytest

import synth
from tests.gpu_util import Lattice, coarse_from_bundle, coarse_to_bundle, relerr, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [(4, 4, 4, 4), (8, 8, 8, 8)])
@pytest.mark.parametrize("nv,nsys", [(1, 1), (1, 33), (6, 8), (8, 9), (10, 16), (13, 17), (24, 8), (24, 33), (28, 1), (32, 9), (32, 16),
                                     (32, 48)])
def test_fp16_coarse_operator(L, nv, nsys):
    torch = torch_cuda()
    lat = Lattice(L, synth.gauge_field(L, 0.3, seed=3), 0.125, 1.0)
    try:
        T = lat.T
        tv = synth.gaussian_spinors(L, nv, seed=5).astype(np.complex64)
        p = T.setup_params(nv=nv, agg=(2, 2, 2, 2), sap_block=(2, 2, 2, 2))
        T.tmamg_setup_from_vectors(lat.ctx, p, torch.from_numpy(tv.view(np.float32).copy()).cuda())
        Vc, nc = int(np.prod(L)) // 16, 2 * nv
        x = synth.complex_normal(7, 1, (nsys, Vc, nc))
        mu = np.linspace(-0.2, 0.3, nsys)
        xb = torch.from_numpy(coarse_to_bundle(x, nc, Vc)).cuda()
        out = {}
        for prec in (32, 16):
            yb = lat.coarse_buffer(nsys)
            T.tmamg_coarse_apply(lat.ctx, 1, xb, yb, nsys, mu, prec)
            torch.cuda.synchronize()
            out[prec] = coarse_from_bundle(yb.cpu().numpy(), nsys, nc, Vc)
        for n in range(nsys):
            assert relerr(out[16][n], out[32][n]) <= 2e-3, n
    finally:
        lat.close()
