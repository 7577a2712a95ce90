"""Restriction and prolongation at the edges of their tilings, against the dense P.

P is taken column by column from the prolongation of unit vectors (one system each) and checked to be
orthonormal; restriction and prolongation of random vectors are then compared with the dense products.
Row counts around the groups of eight, system counts around the tile groups and the largest chunk, and a
level-2 transfer whose K = nv1 x 3 is odd. Tolerance as for the other FP32 components: 2e-5."""
import numpy as np
import pytest

import synth
from tests.gpu_util import Lattice, coarse_from_bundle, coarse_to_bundle, relerr, torch_cuda

pytestmark = pytest.mark.gpu
TOL32 = 2e-5


def _dense(prolong, nc, Vc, batch=64):
    """[parent entries, Vc * nc] columns of P from unit coarse vectors (site-major)"""
    cols = []
    n = Vc * nc
    for k0 in range(0, n, batch):
        m = min(batch, n - k0)
        e = np.zeros((m, n), dtype=complex)
        e[np.arange(m), k0 + np.arange(m)] = 1.0
        cols.append(prolong(e.reshape(m, Vc, nc)).reshape(m, -1).T)
    return np.concatenate(cols, axis=1)


@pytest.mark.parametrize("nv,nsys", [(1, 1), (3, 4), (8, 2), (9, 3), (17, 9), (24, 24), (24, 33), (32, 40), (32, 43)])
def test_transfers_against_dense_p(nv, nsys):
    torch = torch_cuda()
    L = (8, 4, 4, 4)
    lat = Lattice(L, synth.gauge_field(L, 0.3, seed=3), 0.125, 1.0)
    try:
        T = lat.T
        tv = synth.gaussian_spinors(L, nv, seed=5).astype(np.complex64)
        p = T.setup_params(nv=nv, agg=(4, 4, 4, 4), sap_block=(4, 2, 2, 2))
        T.tmamg_setup_from_vectors(lat.ctx, p, torch.from_numpy(tv.view(np.float32).copy()).cuda())
        Vc, nc = 2, 2 * nv

        def prolong(xc):
            n = xc.shape[0]
            cb = torch.from_numpy(coarse_to_bundle(xc, nc, Vc)).cuda()
            fb = torch.full((T.tmamg_bundle_bytes(lat.ctx, n, 32) // 4,), 7.0, device="cuda")
            T.tmamg_prolong(lat.ctx, 1, cb, fb, n)
            return lat.from_fine_bundle(fb, n)

        P = _dense(prolong, nc, Vc)
        assert np.abs(P.conj().T @ P - np.eye(Vc * nc)).max() < TOL32
        x = synth.gaussian_spinors(L, nsys, seed=6)
        cb = lat.coarse_buffer(nsys)
        T.tmamg_restrict(lat.ctx, 1, lat.fine_bundle(x), cb, nsys)
        torch.cuda.synchronize()
        got = coarse_from_bundle(cb.cpu().numpy(), nsys, nc, Vc)
        want = (P.conj().T @ x.astype(np.complex64).reshape(nsys, -1).T).T.reshape(nsys, Vc, nc)
        for n in range(nsys):
            assert relerr(got[n], want[n]) <= TOL32, n
        xc = synth.gaussian_coarse((2, 1, 1, 1), nsys, nv, seed=9).reshape(nsys, Vc, nc)
        up = prolong(xc).reshape(nsys, -1)
        for n in range(nsys):
            assert relerr(up[n], P @ xc[n].ravel()) <= TOL32, n
    finally:
        lat.close()


A16, A8, S16 = (16, 16, 8, 8), (16, 8, 8, 8), (16, 16, 16, 32)


@pytest.mark.parametrize("L,agg,nv,nsys", [
    (A8, (2, 2, 2, 2), 1, 1), (A8, (2, 2, 2, 2), 8, 24), (A8, (2, 2, 2, 2), 9, 12), (A8, (2, 2, 2, 2), 9, 13),
    (A8, (2, 2, 2, 2), 32, 5), (A8, (2, 2, 2, 2), 4, 25), (A8, (4, 2, 2, 2), 24, 12), (A8, (4, 2, 2, 2), 24, 14),
    (A8, (4, 2, 2, 2), 7, 4), (A16, (4, 4, 2, 2), 8, 11), (A16, (4, 4, 2, 2), 9, 3), (A16, (4, 4, 2, 2), 5, 14),
    (A8, (2, 2, 1, 1), 11, 7), (A8, (4, 4, 2, 2), 8, 3), (A16, (4, 4, 4, 2), 3, 8), (S16, (4, 4, 4, 2), 3, 5)])
def test_transfers_with_short_sums(L, agg, nv, nsys):
    """The forms for small aggregates, and the ones beside them: few aggregates, many outputs, longer sums.

    A coarse unit vector on every aggregate at once brings up one column of all their blocks of P."""
    torch = torch_cuda()
    lat = Lattice(L, synth.gauge_field(L, 0.3, seed=3), 0.125, 1.0)
    try:
        T = lat.T
        tv = synth.gaussian_spinors(L, nv, seed=5).astype(np.complex64)
        block = tuple(2 if v == 8 else 4 for v in L)
        p = T.setup_params(nv=nv, agg=agg, sap_block=block)
        T.tmamg_setup_from_vectors(lat.ctx, p, torch.from_numpy(tv.view(np.float32).copy()).cuda())
        Lc = tuple(L[d] // agg[d] for d in range(4))
        Vc, nc = int(np.prod(Lc)), 2 * nv

        def prolong(xc):
            n = xc.shape[0]
            cb = torch.from_numpy(coarse_to_bundle(xc, nc, Vc)).cuda()
            fb = torch.full((T.tmamg_bundle_bytes(lat.ctx, n, 32) // 4,), 7.0, device="cuda")
            T.tmamg_prolong(lat.ctx, 1, cb, fb, n)
            return by_aggregate(lat.from_fine_bundle(fb, n))

        def by_aggregate(x):
            """[n, fine...] -> [n, Vc, 2, K]"""
            n = x.shape[0]
            x = x.reshape(n, Lc[3], agg[3], Lc[2], agg[2], Lc[1], agg[1], Lc[0], agg[0], 2, 6)
            return x.transpose(0, 1, 3, 5, 7, 9, 2, 4, 6, 8, 10).reshape(n, Vc, 2, -1)

        unit = np.zeros((nc, Vc, nc), dtype=complex)
        for j in range(nc):
            unit[j, :, j] = 1.0
        P = prolong(unit)
        up, down = P[:nv], P[nv:]  # chirality 0, then 1
        assert np.all(up[:, :, 1] == 0) and np.all(down[:, :, 0] == 0)
        P = np.stack([up[:, :, 0], down[:, :, 1]])  # [2, nv, Vc, K]
        gram = np.einsum("cjak,clak->acjl", P.conj(), P)
        assert np.abs(gram - np.eye(nv)).max() < TOL32
        x = synth.gaussian_spinors(L, nsys, seed=6).astype(np.complex64)
        cb = lat.coarse_buffer(nsys)
        T.tmamg_restrict(lat.ctx, 1, lat.fine_bundle(x), cb, nsys)
        torch.cuda.synchronize()
        got = coarse_from_bundle(cb.cpu().numpy(), nsys, nc, Vc)
        want = np.einsum("cjak,nack->nacj", P.conj(), by_aggregate(x), optimize=True).reshape(nsys, Vc, nc)
        xc = synth.gaussian_coarse(Lc, nsys, nv, seed=9).reshape(nsys, Vc, nc)
        gotup = prolong(xc)
        wantup = np.einsum("cjak,nacj->nack", P, xc.reshape(nsys, Vc, 2, nv), optimize=True)
        for n in range(nsys):
            assert relerr(got[n], want[n]) <= TOL32, n
            assert relerr(gotup[n], wantup[n]) <= TOL32, n
    finally:
        lat.close()


@pytest.mark.parametrize("nsys", [1, 6, 19])
def test_level_two_transfers_with_odd_k(nsys):
    torch = torch_cuda()
    L = (12, 4, 4, 4)
    nv, nv2 = 5, 7  # K = 5 x 3 per chirality: rows of P2 on 8-byte boundaries only
    lat = Lattice(L, synth.gauge_field(L, 0.3, seed=3), 0.125, 1.0)
    try:
        T = lat.T
        p = T.setup_params(levels=3, nv=nv, nv2=nv2, agg=(4, 4, 4, 4), agg2=(3, 1, 1, 1), sap_block=(2, 2, 2, 2))
        tv = np.concatenate([synth.gaussian_spinors(L, nv, seed=5).ravel(),
                             synth.gaussian_coarse((3, 1, 1, 1), nv2, nv, seed=7).ravel()]).astype(np.complex64)
        T.tmamg_setup_from_vectors(lat.ctx, p, torch.from_numpy(tv.view(np.float32).copy()).cuda())
        nc1, nc2 = 2 * nv, 2 * nv2

        def prolong(xc):
            n = xc.shape[0]
            cb = torch.from_numpy(coarse_to_bundle(xc, nc2, 1)).cuda()
            fb = lat.coarse_buffer(n, 1)
            T.tmamg_prolong(lat.ctx, 2, cb, fb, n)
            torch.cuda.synchronize()
            return coarse_from_bundle(fb.cpu().numpy(), n, nc1, 3)

        P = _dense(prolong, nc2, 1)
        assert np.abs(P.conj().T @ P - np.eye(nc2)).max() < TOL32
        x = synth.gaussian_coarse((3, 1, 1, 1), nsys, nv, seed=8).reshape(nsys, 3, nc1)
        cb = lat.coarse_buffer(nsys, 2)
        T.tmamg_restrict(lat.ctx, 2, torch.from_numpy(coarse_to_bundle(x, nc1, 3)).cuda(), cb, nsys)
        torch.cuda.synchronize()
        got = coarse_from_bundle(cb.cpu().numpy(), nsys, nc2, 1)
        for n in range(nsys):
            assert relerr(got[n].ravel(), P.conj().T @ x[n].ravel()) <= TOL32, n
    finally:
        lat.close()
