"""Performance cases of the tmamg library: what its users have it do, through its public entry points.

A case is a dict of plain values. listed() gives the fixed ones, draw(rng) another one from the same
ranges, prepare(case, seed) the inputs and the context that a program holds before the call, run(state)
one pass, work(case) the bytes and operations a pass cannot do without, exact(case, seed) the result in
64-bit torch arithmetic written here from the operator's definition (include/tmamg.h).

The lattices, system counts and parameters are those of bench.py's workloads (16^3x32 with 12 point
sources, 24^3x48 multi-shift, 32^3x64 with 8 right-hand sides, 40^3x80 with 16 systems), of the tuning
lattice 8^3x16 and of the tests, with ragged ones between them.
"""
import math

import numpy as np
import torch

from paper_2201_03872_gb300 import tmamg as T

KAPPA = 0.1279
EPS = 0.25  # links exp(i eps H), as in the workloads
NV = 24


def _case(kind, L, nsys, **kw):
    c = {"kind": kind, "Lx": L[0], "Ly": L[1], "Lz": L[2], "Lt": L[3], "nsys": nsys}
    c.update(kw)
    return c


def listed():
    def named(name, c):
        return dict(c, name=name)

    return [
        # the fine operator on one system of the small tuning lattice: the latency of one call
        named("stencil32 8x16 n1", _case("dirac", (8, 8, 8, 16), 1, prec=32)),
        # the operator at the size of the largest workload: 16 systems (4 rhs x 4 masses)
        named("stencil32 40x80 n16", _case("dirac", (40, 40, 40, 80), 16, prec=32)),
        # the FP64 operator (outer residuals, checks of solutions), 12 sources of a propagator
        named("stencil64 24x48 n12", _case("dirac", (24, 24, 24, 48), 12, prec=64)),
        # an operator application on a program's own fields (pack, stencil, unpack): ragged extents, odd count
        named("apply32 ragged n5", _case("apply", (20, 12, 28, 44), 5, prec=32)),
        # non-degenerate doublet operator: the 12 sources as 6 flavour pairs
        named("doublet32 16x32 n12", _case("doublet", (16, 16, 16, 32), 12, prec=32)),
        # the smoother as the solver applies it on the precision-form lattice
        named("sap 16x32 n12", _case("sap", (16, 16, 16, 32), 12, bx=4, by=4, bz=4, bt=4, cycles=2, steps=4)),
        # the smoother on a production lattice, 8 right-hand sides
        named("sap 32x64 n8", _case("sap", (32, 32, 32, 64), 8, bx=4, by=4, bz=4, bt=4, cycles=2, steps=4)),
        # transfers between the fine and the first coarse level: the multi-shift workload's 40 systems down,
        # the 16 systems of the largest workload up
        named("restrict 24x48 n40", _case("restrict", (24, 24, 24, 48), 40, nv=NV)),
        named("prolong 24x48 n16", _case("prolong", (24, 24, 24, 48), 16, nv=NV)),
        # the first coarse level's operator (the middle level of a three-level solve)
        named("coarse16 32x64 n16", _case("coarse", (32, 32, 32, 64), 16, nv=NV, cprec=16)),
        # whole solves: a propagator (12 point sources, two levels) and 4 noise sources x 4 masses (three levels)
        named("solve 16x32 n12", _case("solve", (16, 16, 16, 32), 12, levels=2, nshift=1, source="point")),
        named("solve 24x48 4x4", _case("solve", (24, 24, 24, 48), 16, levels=3, nshift=4, source="z2")),
    ]


def _extents(rng, lo, hi, step):
    """Four extents, multiples of step, whose volume is spread over the logarithm of [lo, hi] (sites)."""
    while True:
        v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        side = v ** 0.25
        L = [max(step, int(round(side * math.exp(rng.uniform(-0.4, 0.4)) / step)) * step) for _ in range(3)]
        L.append(max(step, int(round(v / (L[0] * L[1] * L[2]) / step)) * step))
        if lo <= L[0] * L[1] * L[2] * L[3] <= hi and max(L) <= 128:
            return tuple(L)


def _count(rng, hi):
    return max(1, min(hi, int(round(math.exp(rng.uniform(0.0, math.log(hi + 0.49)))))))


def draw(rng):
    kind = rng.choice(["dirac", "dirac", "apply", "doublet", "sap", "sap", "restrict", "prolong", "coarse", "solve"])
    if kind in ("dirac", "apply"):
        prec = rng.choice([32, 32, 64])
        L = _extents(rng, 2048, 600000, 2)
        return _case(kind, L, _count(rng, 40 if kind == "dirac" and prec == 32 else 16), prec=prec)
    if kind == "doublet":
        L = _extents(rng, 2048, 600000, 2)
        return _case(kind, L, 2 * _count(rng, 10), prec=32)
    if kind == "sap":
        b = rng.choice([(4, 4, 4, 4), (4, 4, 4, 4), (8, 4, 4, 2), (4, 4, 2, 4), (2, 2, 2, 2)])
        L = _extents(rng, 4096, 600000, 16 if b[0] == 8 else 8)
        return _case(kind, L, _count(rng, 24), bx=b[0], by=b[1], bz=b[2], bt=b[3], cycles=rng.choice([1, 2, 2, 3]),
                     steps=rng.choice([3, 4, 4, 6]))
    if kind in ("restrict", "prolong", "coarse"):
        L = _extents(rng, 8192, 600000, 4)
        c = _case(kind, L, _count(rng, 40), nv=rng.choice([8, 12, 16, 20, 24, 24, 32]))
        if kind == "coarse":
            c["cprec"] = rng.choice([16, 16, 16, 32])
        return c
    L = _extents(rng, 4096, 140000, 8)
    levels = rng.choice([2, 2, 3])
    nshift = rng.choice([1, 1, 2, 4])
    return _case("solve", L, nshift * _count(rng, 12 // nshift), levels=levels, nshift=nshift,
                 source=rng.choice(["point", "z2"]))


# ------------------------------------------------------------------ inputs
def _dims(case):
    return case["Lx"], case["Ly"], case["Lz"], case["Lt"]


def _volume(case):
    L = _dims(case)
    return L[0] * L[1] * L[2] * L[3]


def _masses(n):
    return np.array([0.005]) if n == 1 else 1.5e-3 * (0.05 / 1.5e-3) ** (np.arange(n) / (n - 1))


def _generator(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + stream) % (1 << 62))
    return g


def _gauge(case, seed):
    """SU(3) links near exp(i EPS H), H Gaussian traceless Hermitian (second order, then reunitarised by
    rows): complex128 [Lt, Lz, Ly, Lx, 4, 3, 3]."""
    n = 4 * _volume(case)
    g = _generator(seed, 1)

    def normal():
        return torch.randn(n, dtype=torch.float64, device="cuda", generator=g) * math.sqrt(0.5)

    d = [normal() for _ in range(3)]
    tr = (d[0] + d[1] + d[2]) / 3.0
    H = {(i, i): torch.complex(d[i] - tr, torch.zeros_like(tr)) for i in range(3)}
    for i, j in ((0, 1), (0, 2), (1, 2)):
        z = torch.complex(normal(), normal()) * math.sqrt(0.5)
        H[i, j], H[j, i] = z, z.conj()
    rows = []
    for i in range(2):
        rows.append([(1.0 if i == j else 0.0) + 1j * EPS * H[i, j]
                     - 0.5 * EPS * EPS * sum(H[i, k] * H[k, j] for k in range(3)) for j in range(3)])
    del H, d, tr

    def unit(r):
        s = torch.rsqrt(sum(c.real * c.real + c.imag * c.imag for c in r))
        return [c * s for c in r]

    r0 = unit(rows[0])
    dot = sum(a.conj() * b for a, b in zip(r0, rows[1]))
    r1 = unit([b - dot * a for a, b in zip(r0, rows[1])])
    r2 = [(r0[(k + 1) % 3] * r1[(k + 2) % 3] - r0[(k + 2) % 3] * r1[(k + 1) % 3]).conj() for k in range(3)]
    U = torch.stack([c.resolve_conj() for c in r0 + r1 + r2], dim=-1)
    Lx, Ly, Lz, Lt = _dims(case)
    return U.view(Lt, Lz, Ly, Lx, 4, 3, 3)


def _fields(case, n, seed, stream, dtype):
    """n complex Gaussian spinor fields [n, V, 12] with unit variance per complex component."""
    g = _generator(seed, stream)
    f = torch.float32 if dtype == torch.complex64 else torch.float64
    return torch.view_as_complex(torch.randn(n, _volume(case), 12, 2, dtype=f, device="cuda", generator=g)
                                 * math.sqrt(0.5))


def _coarse_sites(case):
    return _volume(case) // 256


def _coarse_fields(case, seed):
    """nsys complex Gaussian vectors of the first coarse level, complex64 [nsys, Vc, 2 nv]."""
    g = _generator(seed, 4)
    shape = (case["nsys"], _coarse_sites(case), 2 * case["nv"], 2)
    return torch.view_as_complex(torch.randn(shape, dtype=torch.float32, device="cuda", generator=g) * math.sqrt(0.5))


def _to_bundle(x, t):
    """[nsys, nsite, ncomp] complex -> bundle [ntile, ncomp, nsite, 2, t] real of the same precision."""
    n, sites, comps = x.shape
    nt = (n + t - 1) // t
    b = torch.zeros((nt * t, comps, sites, 2), dtype=x.real.dtype, device=x.device)
    for k in range(n):
        b[k] = torch.view_as_real(x[k].transpose(0, 1).contiguous())
    return b.view(nt, t, comps, sites, 2).permute(0, 2, 3, 4, 1).contiguous()


def _sources(case, seed):
    """Right-hand sides of a solve, complex128 [nrhs, V, 12]."""
    n, V = case["nsys"] // case["nshift"], _volume(case)
    if case["source"] == "point":
        b = torch.zeros((n, V, 12), dtype=torch.complex128, device="cuda")
        site = int(np.random.RandomState(seed % (1 << 31)).randint(V))
        for k in range(n):
            b[k, site, k % 12] = 1.0
        return b
    g = _generator(seed, 5)
    s = torch.randint(0, 2, (n, V, 12, 2), device="cuda", generator=g).to(torch.float64)
    return torch.view_as_complex((2.0 * s - 1.0) * math.sqrt(0.5))


class _State:
    """A context with its operator, and the buffers of one case."""

    def __init__(self, case, seed):
        self.case, self.n = case, case["nsys"]
        self.ctx = T.tmamg_create(_dims(case), -1, torch.cuda.current_stream().cuda_stream)
        U = _gauge(case, seed)
        T.tmamg_load_gauge(self.ctx, U)
        T.tmamg_set_operator(self.ctx, KAPPA, 1.0)
        torch.cuda.current_stream().synchronize()

    def fine_bundle(self, x, prec):
        b = self.empty(T.tmamg_bundle_bytes(self.ctx, x.shape[0], prec), prec)
        T.tmamg_pack(self.ctx, x, b, x.shape[0], prec)
        torch.cuda.current_stream().synchronize()
        return b

    @staticmethod
    def empty(nbytes, prec=32):
        dt = torch.float32 if prec == 32 else torch.float64
        return torch.zeros(nbytes // (prec // 8), dtype=dt, device="cuda")

    def __del__(self):
        ctx, self.ctx = getattr(self, "ctx", None), None
        if ctx:
            T.tmamg_destroy(ctx)


def _setup(case, **kw):
    block = 4 if all(v % 8 == 0 or v == 4 for v in _dims(case)) else 2  # an even number of blocks per dimension
    return T.setup_params(agg=(4, 4, 4, 4), sap_block=(block,) * 4, sap_cycles=2, nv2=32, **kw)


def _solve_params(case):
    # the workloads' solver settings; solutions to 1e-12, two digits below the usual goal
    common = dict(tol=1e-12, max_outer=60, coarse_restart=40, coarse_maxiter=400, sap_cycles=2, sap_mr_steps=4)
    if case["levels"] == 3:
        return T.solve_params(restart=5, inner_cycles=4, coarse_tol=0.2, mid_tol=7e-2, mid_restart=10, mid_maxiter=50,
                              mid_smooth=3, **common)
    return T.solve_params(restart=20, coarse_tol=0.1, **common)


def prepare(case, seed):
    kind = case["kind"]
    s = _State(case, seed)
    n = case["nsys"]
    s.mu = _masses(n)
    if kind in ("dirac", "doublet"):
        prec = case["prec"]
        x = _fields(case, n, seed, 2, torch.complex64 if prec == 32 else torch.complex128)
        s.x = s.fine_bundle(x, prec)
        s.y = torch.zeros_like(s.x)
        if kind == "doublet":
            s.mu, s.eps = _masses(n // 2), 2.0 / 3.0 * _masses(n // 2)
    elif kind == "apply":
        s.x = _fields(case, n, seed, 2, torch.complex64 if case["prec"] == 32 else torch.complex128)
        s.y = torch.zeros_like(s.x)
    elif kind == "sap":
        s.r0 = s.fine_bundle(_fields(case, n, seed, 2, torch.complex64), 32)
        s.r, s.e = torch.empty_like(s.r0), torch.zeros_like(s.r0)
        s.block = (case["bx"], case["by"], case["bz"], case["bt"])
    elif kind in ("restrict", "prolong", "coarse"):
        tv = _fields(case, case["nv"], seed, 3, torch.complex64)
        T.tmamg_setup_from_vectors(s.ctx, _setup(case, nv=case["nv"]), tv)
        del tv
        coarse = s.empty(T.tmamg_coarse_bundle_bytes(s.ctx, 1, n))
        if kind == "restrict":
            s.x, s.y = s.fine_bundle(_fields(case, n, seed, 2, torch.complex64), 32), coarse
        else:
            s.x = _to_bundle(_coarse_fields(case, seed), 2)
            s.y = s.empty(T.tmamg_bundle_bytes(s.ctx, n, 32)) if kind == "prolong" else coarse
    else:
        p = _setup(case, levels=case["levels"], nv=NV, sap_mr_steps=6, setup_iters=20, seed=seed + 1)
        T.tmamg_setup(s.ctx, p)
        s.b = _sources(case, seed)
        s.x = torch.zeros((n,) + tuple(s.b.shape[1:]), dtype=torch.complex128, device="cuda")
        s.mu = _masses(case["nshift"])
        s.params = _solve_params(case)
    return s


def run(s):
    c, kind = s.case, s.case["kind"]
    if kind == "dirac":
        T.tmamg_dirac(s.ctx, s.x, s.y, s.n, s.mu, c["prec"])
    elif kind == "apply":
        T.tmamg_apply(s.ctx, s.x, s.y, s.n, s.mu, c["prec"])
    elif kind == "doublet":
        T.tmamg_dirac_doublet(s.ctx, s.x, s.y, s.n // 2, s.mu, s.eps, c["prec"])
    elif kind == "sap":
        s.r.copy_(s.r0)  # the smoother consumes its residual
        T.tmamg_sap(s.ctx, s.r, s.e, s.n, s.mu, s.block, c["cycles"], c["steps"])
        return {"e": s.e, "r": s.r}
    elif kind == "restrict":
        T.tmamg_restrict(s.ctx, 1, s.x, s.y, s.n)
    elif kind == "prolong":
        T.tmamg_prolong(s.ctx, 1, s.x, s.y, s.n)
    elif kind == "coarse":
        T.tmamg_coarse_apply(s.ctx, 1, s.x, s.y, s.n, s.mu, c["cprec"])
    else:
        T.tmamg_solve(s.ctx, s.b, s.n // c["nshift"], s.mu, c["nshift"], s.x, 1, s.params)
        return s.x
    return s.y


# ------------------------------------------------------------------ what a pass cannot do without
FLOPS_SITE = 1944  # one operator application per site and system: 8 hops, clover blocks, twist


def work(case):
    V, n, kind = _volume(case), case["nsys"], case["kind"]
    field = V * 96 * n  # one FP32 vector per system
    if kind in ("dirac", "apply", "doublet"):
        es = case["prec"] // 8
        return {"bytes": V * (144 + 48 * n) * es, "flops": FLOPS_SITE * V * n}
    if kind == "sap":
        # links and clover, r in and out, e out; per cycle every site takes `steps` block products and one face
        # update (the crossing hops: a quarter of the hops at 4^4 blocks)
        return {"bytes": V * 576 + 3 * field, "flops": case["cycles"] * (case["steps"] * 0.8 + 0.2) * FLOPS_SITE * V * n}
    if kind in ("restrict", "prolong"):
        nv = case["nv"]
        return {"bytes": V * 96 * nv + field + _coarse_sites(case) * 16 * nv * n, "flops": 8 * 12 * nv * V * n}
    if kind == "coarse":
        nc, Vc = 2 * case["nv"], _coarse_sites(case)
        return {"bytes": Vc * (9 * nc * nc * (4 if case["cprec"] == 16 else 8) + 16 * nc * n), "flops": 72 * nc * nc * Vc * n}
    # a solve: both copies of the operator, the transfer vectors, sources in, solutions out; no count of iterations
    # is essential, so the operations are those of one FP64 residual
    return {"bytes": V * (144 * 12 + 96 * NV + 192 * (n // case["nshift"] + n)), "flops": FLOPS_SITE * V * n}


# ------------------------------------------------------------------ the same in 64 bits, by torch
# chiral basis: gamma_k = [[0, -i s_k], [i s_k, 0]], gamma_4 = [[0, 1], [1, 0]]
_GAMMA = np.zeros((4, 4, 4), dtype=complex)
for _k, _s in enumerate(([[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]])):
    _GAMMA[_k, :2, 2:] = -1j * np.array(_s)
    _GAMMA[_k, 2:, :2] = 1j * np.array(_s)
_GAMMA[3, :2, 2:] = _GAMMA[3, 2:, :2] = np.eye(2)


def _spin(m, x):
    """m x on the spin index of x [..., 4, 3], m a 4x4 matrix with one entry per row."""
    col = [int(np.nonzero(m[a])[0][0]) for a in range(4)]
    return torch.stack([x[..., col[a], :] * complex(m[a, col[a]]) for a in range(4)], dim=-2)


def _mm(a, b):
    return (a.unsqueeze(-1) * b.unsqueeze(-3)).sum(-2)


def _dag(a):
    return a.conj().transpose(-1, -2)


def _mv(u, x):
    """u [..., 3, 3] on the colours of x [..., 4, 3]"""
    return (u.unsqueeze(-3) * x.unsqueeze(-2)).sum(-1)


class _Operator:
    def __init__(self, case, seed):
        self.L = _dims(case)
        Lx, Ly, Lz, Lt = self.L
        self.U = _gauge(case, seed)
        self.shape = (Lt, Lz, Ly, Lx, 4, 3)
        self.g5 = torch.tensor([1.0, 1.0, -1.0, -1.0], dtype=torch.float64, device="cuda").view(4, 1)
        U = [self.U[..., nu, :, :] for nu in range(4)]

        def up(a, nu):
            return torch.roll(a, -1, 3 - nu)

        def down(a, nu):
            return torch.roll(a, 1, 3 - nu)

        self.F = []  # (sigma_{mu nu}, F_{mu nu}) for mu < nu, F from the four plaquettes around the site
        for m in range(4):
            for v in range(m + 1, 4):
                mv = _mm(U[m], up(U[v], m))            # U_m(s) U_v(s+m)
                vm = _mm(U[v], up(U[m], v))            # U_v(s) U_m(s+v)
                q = _mm(mv, _dag(vm))                  # s -> s+m -> s+m+v -> s+v -> s
                # s -> s+v -> s+v-m -> s-m -> s: U_v(s) [U_v(s-m) U_m(s-m+v)]^+ U_m(s-m)
                q = q + _mm(_mm(U[v], _dag(down(vm, m))), down(U[m], m))
                # s -> s-m -> s-m-v -> s-v -> s
                q = q + _mm(_dag(down(down(vm, m), v)), down(down(mv, m), v))
                # s -> s-v -> s-v+m -> s+m -> s: U_v(s-v)^+ [U_m(s-v) U_v(s-v+m)] U_m(s)^+
                q = q + _mm(_mm(_dag(down(U[v], v)), down(mv, v)), _dag(U[m]))
                del mv, vm
                sig = 0.5j * (_GAMMA[m] @ _GAMMA[v] - _GAMMA[v] @ _GAMMA[m])
                self.F.append((sig, 0.125 * (q - _dag(q))))
                del q

    def local(self, x, mu):
        y = x * (0.5 / KAPPA) + 1j * mu * self.g5 * x
        for sig, F in self.F:  # (i/4) sum over mu, nu = (i/2) sum over mu < nu
            y += _spin(0.5j * sig, _mv(F, x))
        return y

    def hops(self, x, keep=None):
        """-1/2 sum over the hops of x [Lt, Lz, Ly, Lx, 4, 3]; keep(nu): mask [Lt, Lz, Ly, Lx, 1, 1] of the sites whose
        forward hop in direction nu counts (and with it the backward hop along the same link)."""
        y = torch.zeros_like(x)
        for nu in range(4):
            ax = 3 - nu
            U = self.U[..., nu, :, :]
            w = None if keep is None else keep(nu)
            f = torch.roll(x, -1, ax)
            if nu == 3:
                f[-1] *= -1.0
            f = _mv(U, f - _spin(_GAMMA[nu], f))
            if w is not None:
                f = f * w
            y += f
            b = _mv(_dag(U), x + _spin(_GAMMA[nu], x))
            if w is not None:
                b = b * w
            b = torch.roll(b, 1, ax)
            if nu == 3:
                b[0] *= -1.0
            y += b
        return -0.5 * y

    def apply(self, x, mu):
        """x [V, 12] -> D(mu) x [V, 12]"""
        v = x.to(torch.complex128).view(self.shape)
        return (self.local(v, mu) + self.hops(v)).view(x.shape[0], 12)


def _bundle_of(case, fields, t):
    """[n][V, ncomp] -> FP64 bundle, filled one system at a time"""
    n = case["nsys"]
    nt = (n + t - 1) // t
    out = None
    for k, x in enumerate(fields):
        if out is None:
            out = torch.zeros((nt, x.shape[1], x.shape[0], 2, t), dtype=torch.float64, device="cuda")
        out[k // t, :, :, :, k % t] = torch.view_as_real(x.transpose(0, 1).contiguous())
    return out.view(-1)


def _sap_exact(case, seed):
    op = _Operator(case, seed)
    L, bs = op.L, (case["bx"], case["by"], case["bz"], case["bt"])
    nb = [L[k] // bs[k] for k in range(4)]
    coord = [torch.arange(L[k], device="cuda").view([-1 if 3 - k == a else 1 for a in range(4)] + [1, 1]) for k in range(4)]
    parity = sum(coord[k] // bs[k] for k in range(4)) % 2
    parity = parity.expand(L[3], L[2], L[1], L[0], 1, 1)
    inside = [((coord[k] % bs[k]) != bs[k] - 1).to(torch.float64) if nb[k] > 1 else torch.ones(1, device="cuda", dtype=torch.float64)
              for k in range(4)]

    def block_sum(a):  # [Lt, Lz, Ly, Lx] -> its block's sum at every site
        v = a.view(nb[3], bs[3], nb[2], bs[2], nb[1], bs[1], nb[0], bs[0]).sum((1, 3, 5, 7), keepdim=True)
        return v.expand(nb[3], bs[3], nb[2], bs[2], nb[1], bs[1], nb[0], bs[0]).reshape(a.shape)

    def dot(a, b):
        return block_sum((a.conj() * b).sum((-1, -2))).unsqueeze(-1).unsqueeze(-1)

    colours = 1 if all(v == 1 for v in nb) else 2
    mus = _masses(case["nsys"])
    x = _fields(case, case["nsys"], seed, 2, torch.complex64)

    def one(k):
        r = x[k].to(torch.complex128).view(op.shape)
        e = torch.zeros_like(r)
        for cy in range(case["cycles"]):
            for col in range(colours):
                on = (parity == col).to(torch.float64)
                rho = r * on
                d = torch.zeros_like(r)
                for _ in range(case["steps"]):
                    q = op.local(rho, mus[k]) + op.hops(rho, lambda nu: inside[nu])
                    qq = dot(q, q).real
                    alpha = torch.where(qq > 0, dot(q, rho) / torch.where(qq > 0, qq, torch.ones_like(qq)), torch.zeros_like(qq) + 0j)
                    d = d + alpha * rho
                    rho = rho - alpha * q
                e = e + d
                r = r * (1.0 - on) + rho
                if colours == 2 and not (cy == case["cycles"] - 1 and col == 1):
                    r = r - op.hops(d, lambda nu: 1.0 - inside[nu]) * (1.0 - on)
        return e.view(-1, 12), r.view(-1, 12)

    both = [one(k) for k in range(case["nsys"])]
    return {"e": _bundle_of(case, [b[0] for b in both], 2), "r": _bundle_of(case, [b[1] for b in both], 2)}


class _Transfer:
    """P of the first level from the test vectors: orthonormal per 4^4 aggregate and chirality, in their order."""

    def __init__(self, case, seed):
        self.L, self.nv = _dims(case), case["nv"]
        v = torch.stack([self.split(f) for f in _fields(case, self.nv, seed, 3, torch.complex64)], dim=-1)
        c = torch.linalg.cholesky(v.mH @ v)  # v = P c^+: the Gram-Schmidt basis
        self.P = torch.linalg.solve_triangular(c.mH, v, upper=True, left=False)

    def split(self, x):
        """[V, 12] -> [Vc, 2, 256 * 6]: the entries of each aggregate and chirality"""
        a = [v // 4 for v in self.L]
        y = x.to(torch.complex128).view(a[3], 4, a[2], 4, a[1], 4, a[0], 4, 2, 6).permute(0, 2, 4, 6, 8, 1, 3, 5, 7, 9)
        return y.reshape(a[0] * a[1] * a[2] * a[3], 2, 256 * 6)

    def merge(self, y):
        a = [v // 4 for v in self.L]
        x = y.view(a[3], a[2], a[1], a[0], 2, 4, 4, 4, 4, 6).permute(0, 5, 1, 6, 2, 7, 3, 8, 4, 9)
        return x.reshape(-1, 12)

    def down(self, x):
        return (self.P.mH @ self.split(x).unsqueeze(-1)).squeeze(-1).reshape(-1, 2 * self.nv)

    def up(self, xc):
        return self.merge((self.P @ xc.to(torch.complex128).view(-1, 2, self.nv, 1)).squeeze(-1))


def _solve_exact(case, seed):
    """BiCGStab in 64 bits on every (source, mass) at once; None where it does not reach 1e-13 or would take long."""
    if _volume(case) * case["nsys"] > 1700000 or case["nshift"] != 1:
        return None
    op = _Operator(case, seed)
    mu = float(_masses(1)[0])
    b = _sources(case, seed).view((case["nsys"],) + op.shape)
    n = b.shape[0]

    def A(x):
        return torch.stack([op.apply(x[k].reshape(-1, 12), mu).view(op.shape) for k in range(n)])

    def dot(u, v):
        return (u.conj() * v).reshape(n, -1).sum(1).view(n, 1, 1, 1, 1, 1, 1)

    def ratio(u, v):
        return torch.where(v.abs() > 0, u / torch.where(v.abs() > 0, v, torch.ones_like(v)), torch.zeros_like(u))

    x = torch.zeros_like(b)
    bb = dot(b, b).real
    for _ in range(3):  # restarted from the true residual
        r = b - A(x)
        s, p, rho = r.clone(), r.clone(), dot(r, r)
        for it in range(220):
            v = A(p)
            alpha = ratio(rho, dot(s, v))
            x += alpha * p
            r = r - alpha * v
            t = A(r)
            omega = ratio(dot(t, r), dot(t, t))
            x += omega * r
            r = r - omega * t
            new = dot(s, r)
            beta = ratio(new, rho) * ratio(alpha, omega)
            p = r + beta * (p - omega * v)
            rho = new
            if it % 10 == 9 and float((dot(r, r).real / bb).max()) < 1e-28:
                break
        r = b - A(x)
        if float((dot(r, r).real / bb).max()) < 1e-26:
            return x.reshape(n, -1, 12)
    return None


def exact(case, seed):
    kind, n = case["kind"], case["nsys"]
    if kind == "solve":
        return _solve_exact(case, seed)
    if kind == "sap":
        return _sap_exact(case, seed)
    if kind in ("restrict", "prolong", "coarse"):
        P = _Transfer(case, seed)
        if kind == "restrict":
            x = _fields(case, n, seed, 2, torch.complex64)
            return _bundle_of(case, (P.down(x[k]) for k in range(n)), 2)
        xc = _coarse_fields(case, seed)
        if kind == "prolong":
            return _bundle_of(case, (P.up(xc[k]) for k in range(n)), 2)
        op, mu = _Operator(case, seed), _masses(n)  # D_c = P^+ D P
        y = _bundle_of(case, (P.down(op.apply(P.up(xc[k]), mu[k])) for k in range(n)), 2)
        return y
    prec = case["prec"]
    op = _Operator(case, seed)
    x = _fields(case, n, seed, 2, torch.complex64 if prec == 32 else torch.complex128)
    if kind == "apply":
        return torch.stack([op.apply(x[k], m) for k, m in enumerate(_masses(n))])
    if kind == "dirac":
        return _bundle_of(case, (op.apply(x[k], m) for k, m in enumerate(_masses(n))), 2 if prec == 32 else 1)
    mus, out = _masses(n // 2), []
    for q, m in enumerate(mus):
        u, d = x[2 * q].to(torch.complex128), x[2 * q + 1].to(torch.complex128)
        out += [op.apply(u, m) - 2.0 / 3.0 * m * d, op.apply(d, -m) - 2.0 / 3.0 * m * u]
    return _bundle_of(case, out, 2)
