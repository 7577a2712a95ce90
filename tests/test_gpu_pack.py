"""User fields <-> bundles: exact copies at the edges of the 128-site transposition.

Lattices of fewer and more than 128 sites and with a remainder, odd and even system counts (the absent system of
the last FP32 tile is zero), and fields and bundles that start one real past an aligned address."""
import numpy as np
import pytest

import synth
from tests.gpu_util import Lattice, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("L,nsys", [((2, 2, 2, 2), 1), ((4, 4, 4, 2), 2), ((6, 4, 2, 4), 3), ((10, 2, 6, 4), 5), ((4, 4, 4, 6), 4)])
def test_pack_unpack_exact(L, nsys, prec):
    torch = torch_cuda()
    lat = Lattice(L, synth.unit_gauge(L), 0.125, 1.0)
    try:
        T = lat.T
        V, tile = int(np.prod(L)), 2 if prec == 32 else 1
        nt = -(-nsys // tile)
        real = np.float32 if prec == 32 else np.float64
        x = np.random.default_rng(4).standard_normal((nsys, V, 12, 2)).astype(real)
        want = np.zeros((nt * tile, V, 12, 2), dtype=real)
        want[:nsys] = x
        want = want.reshape(nt, tile, V, 12, 2).transpose(0, 3, 2, 4, 1)  # [tile][component][site][re, im][system]
        for off in (0, 1):
            f = torch.zeros(x.size + off, dtype=torch.from_numpy(x).dtype, device="cuda")
            f[off:] = torch.from_numpy(x.ravel()).cuda()
            b = torch.full((want.size + off,), 7.0, dtype=f.dtype, device="cuda")
            T.tmamg_pack(lat.ctx, f[off:], b[off:], nsys, prec)
            torch.cuda.synchronize()
            assert np.array_equal(b[off:].cpu().numpy(), want.ravel())
            back = torch.full((x.size + off + 3,), 7.0, dtype=f.dtype, device="cuda")
            T.tmamg_unpack(lat.ctx, b[off:], back[off:], nsys, prec)
            torch.cuda.synchronize()
            assert np.array_equal(back[off:off + x.size].cpu().numpy(), x.ravel())
            assert (back[off + x.size:] == 7.0).all() and (back[:off] == 7.0).all()
    finally:
        lat.close()
