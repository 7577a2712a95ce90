"""tmamg_apply against its parts (pack, stencil, unpack), bit for bit: the forms that write the user field themselves and
those that do not, sites that do not fill the last 32, one to eight tiles per block, odd system counts, fields one real
past an aligned address, y in place of x, and nothing written beyond the field."""
import numpy as np
import pytest

import synth
from tests.gpu_util import Lattice, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", [0, 1, 2, 3])
@pytest.mark.parametrize("L,nsys", [((2, 2, 2, 2), 1), ((6, 2, 4, 2), 3), ((10, 2, 6, 4), 6), ((4, 4, 4, 4), 11), ((4, 2, 2, 6), 16)])
def test_apply_equals_parts(L, nsys, variant):
    torch = torch_cuda()
    lat = Lattice(L, synth.gauge_field(L, 0.4, seed=6), 0.124, 1.1)
    T = lat.T
    try:
        V = int(np.prod(L))
        x = torch.from_numpy(synth.gaussian_spinors(L, nsys, seed=7).astype(np.complex64).view(np.float32).ravel()).cuda()
        mu = np.linspace(-0.1, 0.2, nsys)
        T.tmamg_autotune_force(variant)
        nb = T.tmamg_bundle_bytes(lat.ctx, nsys, 32) // 4
        xb, yb = (torch.zeros(nb, device="cuda") for _ in range(2))
        T.tmamg_pack(lat.ctx, x, xb, nsys, 32)
        T.tmamg_dirac(lat.ctx, xb, yb, nsys, mu, 32)
        want = torch.empty_like(x)
        T.tmamg_unpack(lat.ctx, yb, want, nsys, 32)
        for off in (0, 1):
            buf = torch.full((x.numel() + off + 5,), 7.0, device="cuda")
            T.tmamg_apply(lat.ctx, x, buf[off:], nsys, mu, 32)
            torch.cuda.synchronize()
            assert torch.equal(buf[off:off + x.numel()], want)
            assert (buf[off + x.numel():] == 7.0).all() and (buf[:off] == 7.0).all()
        T.tmamg_apply(lat.ctx, x, x, nsys, mu, 32)
        torch.cuda.synchronize()
        assert torch.equal(x, want)
    finally:
        T.tmamg_autotune_force(-1)
        lat.close()


@pytest.mark.parametrize("L,nsys", [((4, 4, 4, 4), 1), ((4, 4, 4, 4), 6), ((16, 16, 16, 28), 2), ((16, 16, 16, 28), 3)])
def test_untuned_forms_same_bits(L, nsys):
    """With tuning off: the direct form for one tile and for few sites, else the staged one (from 116736 sites x tiles)."""
    torch = torch_cuda()
    lat = Lattice(L, synth.gauge_field(L, 0.4, seed=6), 0.124, 1.1)
    T = lat.T
    try:
        x = torch.from_numpy(synth.gaussian_spinors(L, nsys, seed=7).astype(np.complex64).view(np.float32).ravel()).cuda()
        xb, mu = lat.fine_bundle(synth.gaussian_spinors(L, nsys, seed=7)), np.linspace(-0.1, 0.2, nsys)
        out = []
        for off in (False, True):
            if off:
                T.tmamg_autotune(0)
            else:
                T.tmamg_autotune_force(1)
            y, f = torch.full_like(xb, 7.0), torch.empty_like(x)
            T.tmamg_dirac(lat.ctx, xb, y, nsys, mu, 32)
            T.tmamg_apply(lat.ctx, x, f, nsys, mu, 32)
            torch.cuda.synchronize()
            out.append((y, f))
            T.tmamg_autotune_force(-1)
        assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    finally:
        T.tmamg_autotune_force(-1)
        T.tmamg_autotune(1)
        lat.close()
