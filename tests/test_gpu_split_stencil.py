"""The FP32 stencil's split form against the direct form, bit for bit: lattices whose sites do not fill the last 32,
one site per direction pair (extent 2: both neighbours are the same site), one to three tiles, more systems than
the kernel takes masses for as values, the antiperiodic boundary and the doublet's coupling. (The direct form is
compared with the oracle elsewhere.)"""
import numpy as np
import pytest

import synth
from tests.gpu_util import Lattice, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,nsys", [((2, 2, 2, 2), 1), ((2, 2, 2, 6), 2), ((6, 2, 4, 2), 3), ((4, 4, 4, 4), 5), ((10, 2, 6, 4), 6), ((4, 4, 4, 4), 34)])
def test_split_form_same_bits(L, nsys):
    torch = torch_cuda()
    lat = Lattice(L, synth.gauge_field(L, 0.4, seed=6), 0.124, 1.1)
    T = lat.T
    try:
        x = lat.fine_bundle(synth.gaussian_spinors(L, nsys, seed=7))
        npair = nsys // 2
        out = []
        for v in (1, 3):
            T.tmamg_autotune_force(v)
            y = torch.full_like(x, 7.0)
            T.tmamg_dirac(lat.ctx, x, y, nsys, np.linspace(-0.1, 0.2, nsys), 32)
            z = torch.full_like(x, 7.0)
            if npair:
                T.tmamg_dirac_doublet(lat.ctx, x, z, npair, np.linspace(0.1, 0.2, npair), np.linspace(0.0, 0.3, npair), 32)
            torch.cuda.synchronize()
            out.append((y.cpu().numpy(), z.cpu().numpy()))
        assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    finally:
        T.tmamg_autotune_force(-1)
        lat.close()


def test_more_tiles_than_a_grid_has_rows():
    # FP32: two systems per tile; a grid's second extent ends at 65535
    torch = torch_cuda()
    L, nsys = (2, 2, 2, 2), 2 * 65535 + 5
    lat = Lattice(L, synth.gauge_field(L, 0.4, seed=6), 0.124, 1.1)
    T = lat.T
    try:
        x = torch.randn(T.tmamg_bundle_bytes(lat.ctx, nsys, 32) // 4, device="cuda")
        mu = np.linspace(-0.1, 0.2, nsys)
        out = []
        for v in (1, 3, -1):
            T.tmamg_autotune_force(v)
            y = torch.full_like(x, 7.0)
            T.tmamg_dirac(lat.ctx, x, y, nsys, mu, 32)
            out.append(y)
        torch.cuda.synchronize()
        valid = torch.ones_like(x, dtype=torch.bool).view(-1, 2)
        valid[-12 * 16 * 2:, 1] = False  # the last tile's padding lane
        valid = valid.view(-1)
        assert torch.equal(out[0][valid], out[1][valid]) and torch.equal(out[0][valid], out[2][valid])
    finally:
        T.tmamg_autotune_force(-1)
        lat.close()
