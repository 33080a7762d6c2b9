"""Workloads of this library as its users run them, for measuring how long each takes.

``listed()`` names them, ``draw(rng)`` gives more of the same ranges, ``prepare(case, seed)``
makes on the GPU what a program has in hand before the call, ``run(state)`` is one call through
the public API, ``work(case)`` the bytes and flops the call cannot do without, and
``exact(case, seed)`` its result in plain 64-bit torch, written from the definitions (no code of
the package).

The kinds of call:

* ``dslash``    the Wilson-Dirac stencil on fields and links in the ABI layout, every storage type,
                full lattice or one parity;
* ``schur``     the even-odd Schur complement (even-odd preconditioning);
* ``vectors``   the smoothed test vectors of one stream of the setup (Eq. 2);
* ``svd``       the streaming chiral SVD of given test vectors into the prolongator (Algorithm 3);
* ``galerkin``  the coarse operator P^dag D P of a given prolongator (Eq. 5), and its export;
* ``solve``     D x = b with a hierarchy that was set up before (many right-hand sides per
                configuration: the usual life of a hierarchy);
* ``step``      setup + coarse operator + solve of one right-hand side (one per configuration);
* ``adjoint``   forward solve and backward (adjoint solve, link-angle gradient) through autograd.

Solves run to a residual of 1e-12, so that x is fixed to better than 1e-9 whatever path the
iteration took.  Results that the library forms in FP32 and hands out in a wider type (test
vectors, singular values of FP32 test vectors) are kept in the type they were formed in.
"""
import math

import torch

from paper_2505_14399_gb300 import api

DEV = "cuda"

ISO = "iso"            # hop weights 1, periodic
ISO_AP = "iso_ap"      # hop weights 1, antiperiodic in t
ANISO_AP = "aniso_ap"  # temporal hop weight 1 / 3.5, antiperiodic in t


def _wbc(case):
    w = (1.0, 1.0, 1.0, 1.0 / 3.5) if case["action"] == ANISO_AP else (1.0, 1.0, 1.0, 1.0)
    bc = (1, 1, 1, 1) if case["action"] == ISO else (1, 1, 1, -1)
    return w, bc


def _dims(case):
    return (case["Lx"], case["Ly"], case["Lz"], case["Lt"])


def _block(case):
    return (case["bx"], case["by"], case["bz"], case["bt"])


def _vol(case):
    return case["Lx"] * case["Ly"] * case["Lz"] * case["Lt"]


def _stencil(kind, name, dims, dtype, nrhs, action, kappa, parity=-1, dagger=False):
    c = dict(kind=kind, Lx=dims[0], Ly=dims[1], Lz=dims[2], Lt=dims[3], dtype=dtype, nrhs=nrhs,
             action=action, kappa=kappa, parity=parity, dagger=dagger)
    return dict(c, name=name) if name else c


def _mg(kind, name, dims, block, k, r, n_s, action, kappa, nrhs=1, schur=0, stream=0):
    c = dict(kind=kind, Lx=dims[0], Ly=dims[1], Lz=dims[2], Lt=dims[3], bx=block[0], by=block[1],
             bz=block[2], bt=block[3], k=k, r=r, n_s=n_s, action=action, kappa=kappa, nrhs=nrhs,
             schur=schur, stream=stream)
    return dict(c, name=name) if name else c


def listed():
    near = 0.1358688963   # 0.995 of the critical value of such links on 16^3x32
    return [
        # the smallest call: latency of one stencil on the FP64 parity lattice
        _stencil("dslash", "dslash_4x4x4x4_c128", (4, 4, 4, 4), "c128", 1, ISO, 0.124),
        # one FP32 stencil on the lattice that one GPU usually holds: a user's own Krylov solver
        _stencil("dslash", "dslash_16x16x16x32_c64", (16, 16, 16, 32), "c64", 1, ISO, near),
        # the largest: twelve right-hand sides (spin x colour sources) on 32^3x64
        _stencil("dslash", "dslash_32x32x32x64_c64_12rhs", (32, 32, 32, 64), "c64", 12, ISO, 0.1338),
        # half storage on the anisotropic lattice, antiperiodic in time
        _stencil("dslash", "dslash_16x16x16x64_bf16", (16, 16, 16, 64), "bf16", 1, ANISO_AP, 0.1621),
        # even-odd preconditioned operator, extents that are no powers of two, three sources
        _stencil("schur", "schur_12x10x14x18_c64_3rhs", (12, 10, 14, 18), "c64", 3, ISO_AP, 0.13),
        # one stream of the setup's test vectors
        _mg("vectors", "vectors_16x16x16x32", (16, 16, 16, 32), (4, 4, 4, 4), 12, 8, 4, ISO, near),
        # the streaming SVD of 32 near-null vectors that the application brings itself
        _mg("svd", "svd_16x16x16x32", (16, 16, 16, 32), (4, 4, 4, 4), 12, 8, 4, ISO, near),
        # the coarse operator, k = 12 on 4^4 aggregates
        _mg("galerkin", "galerkin_16x16x16x32_k12", (16, 16, 16, 32), (4, 4, 4, 4), 12, 8, 4, ISO,
            near),
        # the coarse operator, k = 24 on the anisotropic lattice's 2x2x2x4 aggregates
        _mg("galerkin", "galerkin_16x16x16x64_k24", (16, 16, 16, 64), (2, 2, 2, 4), 24, 16, 4,
            ANISO_AP, 0.1621),
        # a solve near the critical mass on a hierarchy made before (Schur-form smoother)
        _mg("solve", "solve_16x16x16x32", (16, 16, 16, 32), (4, 4, 4, 4), 12, 8, 4, ISO, near,
            schur=1),
        # a new configuration: setup, coarse operator and one solve
        _mg("step", "step_16x16x16x32", (16, 16, 16, 32), (4, 4, 4, 4), 12, 8, 4, ISO, near,
            schur=1),
        # training through the solve: forward, backward to the source and the link angles
        _mg("adjoint", "adjoint_8x8x8x8", (8, 8, 8, 8), (2, 2, 2, 2), 8, 8, 2, ISO, 0.12),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_mg_dims(rng, block, vmax):
    """Extents block x (2 ...) that are even, spread over their logarithm, volume <= vmax."""
    while True:
        dims = []
        for b in block:
            n = _log_int(rng, 2, 12)
            dims.append(b * (n + (b * n) % 2))
        v = dims[0] * dims[1] * dims[2] * dims[3]
        if 256 <= v <= vmax:
            return tuple(dims)


def draw(rng):
    kind = rng.choice(["dslash"] * 4 + ["schur"] + ["vectors"] * 2 + ["svd"] * 2 + ["galerkin"] * 2 +
                      ["solve"] * 2 + ["step"] * 2 + ["adjoint"])
    action = rng.choice([ISO, ISO_AP, ANISO_AP])
    if kind in ("dslash", "schur"):
        parity = rng.choice([-1, -1, 0, 1]) if kind == "dslash" else -1
        even = kind == "schur" or parity >= 0
        while True:
            dims = [_log_int(rng, 3, 40) for _ in range(4)]
            if even:
                dims = [d + d % 2 for d in dims]
            nrhs = rng.choice([1, 1, 2, 3, 5, 8, 12])
            v = dims[0] * dims[1] * dims[2] * dims[3]
            if v * nrhs <= 1 << 22:
                break
        return _stencil(kind, None, dims, rng.choice(["c64", "c64", "c128", "f16", "bf16"]), nrhs,
                        action, round(rng.uniform(0.11, 0.134), 5), parity, rng.random() < 0.25)
    block = rng.choice([(2, 2, 2, 2), (4, 4, 4, 4), (2, 2, 2, 4), (4, 4, 2, 2), (3, 3, 3, 3),
                        (2, 4, 4, 2)])
    rows = 6 * block[0] * block[1] * block[2] * block[3]
    vmax = 1 << 13 if kind == "adjoint" else 1 << 17
    dims = _draw_mg_dims(rng, block, vmax)
    while True:
        k, r, n_s = rng.randint(4, 24), rng.randint(4, 24), rng.randint(1, 4)
        if kind in ("solve", "step", "adjoint"):
            k, r = min(k, 16), min(r, 12)
        if r * n_s >= k and 2 * (k + r) <= rows and k + r <= 48:
            break
    kappa = rng.choice([0.115, 0.12, 0.13, 0.1338])
    if kind in ("solve", "step"):
        return _mg(kind, None, dims, block, k, r, n_s, rng.choice([ISO, ISO_AP]), kappa,
                   nrhs=rng.choice([1, 1, 2, 4]) if kind == "solve" else 1, schur=rng.choice([0, 1]))
    if kind == "adjoint":
        return _mg(kind, None, dims, block, k, r, n_s, rng.choice([ISO, ISO_AP]), min(kappa, 0.12))
    return _mg(kind, None, dims, block, k, r, n_s, action, kappa,
               stream=rng.randrange(n_s) if kind == "vectors" else 0)


# ------------------------------------------------------------------------------------ inputs
def _gauss(g, shape):
    return torch.complex(torch.randn(shape, generator=g, device=DEV, dtype=torch.float64),
                         torch.randn(shape, generator=g, device=DEV, dtype=torch.float64))


def _smooth_links(g, V, eps=0.3):
    """SU(3) links near the identity, complex128 (4, V, 3, 3): exp(i eps H), H traceless
    Hermitian Gaussian, through its Taylor series and a Gram-Schmidt of the rows."""
    out = torch.empty((4, V, 3, 3), device=DEV, dtype=torch.complex128)
    eye = torch.eye(3, device=DEV, dtype=torch.complex128)
    for mu in range(4):
        A = _gauss(g, (V, 3, 3))
        H = 0.5 * (A + A.mH)
        H = H - (torch.einsum("xaa->x", H) / 3)[:, None, None] * eye
        X = (1j * eps) * H
        U = eye.expand(V, 3, 3)
        for n in range(8, 0, -1):     # Horner form of the series
            U = eye + torch.matmul(X, U) / n
        r0 = U[:, 0] / torch.linalg.vector_norm(U[:, 0], dim=1, keepdim=True)
        r1 = U[:, 1] - (r0.conj() * U[:, 1]).sum(1, keepdim=True) * r0
        r1 = r1 / torch.linalg.vector_norm(r1, dim=1, keepdim=True)
        r2 = torch.linalg.cross(r0, r1).conj()
        out[mu] = torch.stack([r0, r1, r2], dim=1)
    return out


_TORCH = {"c128": torch.complex128, "c64": torch.complex64, "f16": torch.float16,
          "bf16": torch.bfloat16}


def _store(x, dtype):
    """complex128 -> the storage type (half types: a trailing (re, im) dimension)."""
    if dtype in ("c128", "c64"):
        return x.to(_TORCH[dtype])
    return torch.view_as_real(x).to(_TORCH[dtype])


def _widen(x):
    """A stored field -> complex128."""
    if x.is_complex():
        return x.to(torch.complex128)
    return torch.view_as_complex(x.to(torch.float64))


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _stencil_inputs(case, seed):
    g = _gen(seed)
    V = _vol(case)
    links = _store(_smooth_links(g, V), case["dtype"])
    n = V if case["kind"] == "dslash" and case["parity"] < 0 else V // 2
    psi = torch.stack([_store(_gauss(g, (n, 4, 3)), case["dtype"]) for _ in range(case["nrhs"])])
    return psi, links


def _mg_inputs(case, seed):
    """What a multigrid program starts from: links, and per kind its sources / test vectors /
    prolongator."""
    g = _gen(seed)
    V = _vol(case)
    links = _smooth_links(g, V)
    if case["kind"] == "svd":
        # test vectors whose tiles have singular values spread over two decades
        m = case["n_s"] * case["r"]
        vec = torch.empty((m, V, 4, 3), device=DEV, dtype=torch.complex64)
        for i in range(m):
            vec[i] = (_gauss(g, (V, 4, 3)) * 10.0 ** (-2.0 * i / max(m - 1, 1))).to(torch.complex64)
        return links, vec
    if case["kind"] == "galerkin":
        # orthonormal tiles (d, 2, k, rows): Gram-Schmidt, twice, of complex Gaussians
        bx, by, bz, bt = _block(case)
        nd = bx * by * bz * bt
        k = case["k"]
        P = _gauss(g, (V // nd * 2, k, 6 * nd))
        for i in range(k):
            v = P[:, i]
            for _ in range(2):
                if i:
                    c = torch.einsum("tir,tr->ti", P[:, :i].conj(), v)
                    v = v - torch.einsum("tir,ti->tr", P[:, :i], c)
            P[:, i] = v / torch.linalg.vector_norm(v, dim=1, keepdim=True)
        return links, P.reshape(V // nd, 2, k, 6 * nd)
    if case["kind"] == "vectors":
        return links, None
    return links, _gauss(g, (case["nrhs"], V, 4, 3))


def _params(case, seed):
    w, bc = _wbc(case)
    return api.params(_dims(case), _block(case), case["kappa"], case["k"], case["r"], case["n_s"],
                      5, _tv_seed(seed), w, bc, setup_dtype="c64", solve_dtype="c64",
                      schur_smoother=case["schur"])


def _tv_seed(seed):
    return 3000 + 7 * int(seed)


def prepare(case, seed):
    s = {"case": case}
    if case["kind"] in ("dslash", "schur"):
        s["psi"], s["links"] = _stencil_inputs(case, seed)
        return s
    s["links"], x = _mg_inputs(case, seed)
    s["p"] = _params(case, seed)
    if case["kind"] == "svd":
        s["vec"] = x
    elif case["kind"] == "galerkin":
        s["h"] = api.Hierarchy(s["links"], s["p"], setup=False)
        s["h"].set_prolongator(x)
    elif case["kind"] == "solve":
        s["b"] = x
        s["h"] = api.Hierarchy(s["links"], s["p"])
        s["h"].coarse_build()
    elif case["kind"] == "step":
        s["b"] = x
    elif case["kind"] == "adjoint":
        s["b"] = x.requires_grad_()
        s["omega"] = torch.zeros((4, _vol(case), 8), device=DEV, dtype=torch.float64,
                                 requires_grad=True)
        s["h"] = api.Hierarchy(s["links"], s["p"])
        s["h"].coarse_build()
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "dslash":
        w, bc = _wbc(case)
        return api.dslash(s["psi"], s["links"], _dims(case), case["kappa"], w, bc,
                          parity=case["parity"], dagger=case["dagger"])
    if kind == "schur":
        w, bc = _wbc(case)
        return api.schur(s["psi"], s["links"], _dims(case), case["kappa"], w, bc,
                         dagger=case["dagger"])
    if kind == "vectors":
        # smoothed in FP32: kept in complex64, as mg_setup_from_vectors takes them
        return api.test_vectors(s["links"], s["p"], case["stream"]).to(torch.complex64)
    if kind == "svd":
        h = api.Hierarchy(s["links"], s["p"], vectors=s["vec"])
        P, sigma = h.prolongator()
        h.close()
        return P, sigma
    if kind == "galerkin":
        s["h"].coarse_build()
        return s["h"].coarse_op()
    if kind == "solve":
        return s["h"].solve(s["b"], tol=1e-12)[0]
    if kind == "step":
        h = api.Hierarchy(s["links"], s["p"])
        h.coarse_build()
        x, _ = h.solve(s["b"], tol=1e-12)
        sigma = h.sigma_history().to(torch.float32)   # of FP32 test vectors
        h.close()
        return x, sigma
    x = api.mg_solve_autograd(s["b"], s["omega"], s["h"], s["links"], tol=1e-12)
    loss = torch.view_as_real(x).square().sum()
    g_b, g_omega = torch.autograd.grad(loss, (s["b"], s["omega"]))
    return x.detach(), g_b, g_omega


# -------------------------------------------------------------------------------------- work
_BYTES = {"c128": 16, "c64": 8, "f16": 4, "bf16": 4}   # of one complex number


def work(case):
    V = _vol(case)
    kind = case["kind"]
    if kind in ("dslash", "schur"):
        e, n = _BYTES[case["dtype"]], case["nrhs"]
        sites = V if kind == "dslash" and case["parity"] < 0 else V // 2
        hops = sites if kind == "dslash" else V
        return {"bytes": e * (24 * sites * n + 36 * V), "flops": 1320 * hops * n}
    k, r, n_s = case["k"], case["r"], case["n_s"]
    links = 16 * 36 * V
    smooth = (1320 * 6 + 48 * 2 * 15 + 96) * V      # D phi, five steps and their projections
    kk, svd = 0, 0
    for _ in range(n_s):
        c = kk + r
        kn = min(c, k)
        svd += 8 * 12 * V * (c * (c + 1) // 2 + c * kn)
        kk = kn
    galerkin = 768 * k * k * V
    d = V // (case["bx"] * case["by"] * case["bz"] * case["bt"])
    opbytes = 16 * 9 * d * 4 * k * k
    pbytes = 16 * 12 * V * k
    # a solve: one K-cycle (restrict, prolong, ten stencils) per decimal digit of the residual
    solve = 12 * (1320 * 10 + 2 * 96 * k) * V * case["nrhs"]
    field = 16 * 12 * V
    if kind == "vectors":
        return {"bytes": links + field * r, "flops": smooth * r}
    if kind == "svd":
        return {"bytes": links + field // 2 * r * n_s + pbytes, "flops": svd}
    if kind == "galerkin":
        return {"bytes": links + pbytes + opbytes, "flops": galerkin}
    if kind == "solve":
        return {"bytes": links + pbytes + 2 * field * case["nrhs"], "flops": solve}
    if kind == "step":
        return {"bytes": links + 2 * field, "flops": smooth * r * n_s + svd + galerkin + solve}
    return {"bytes": links + pbytes + 4 * field + 8 * 32 * V, "flops": 2 * solve + 4000 * V}


# ------------------------------------------------------- the definitions in plain 64-bit torch
def _gammas():
    s = torch.zeros((3, 2, 2), dtype=torch.complex128)
    s[0, 0, 1] = s[0, 1, 0] = 1
    s[1, 0, 1], s[1, 1, 0] = -1j, 1j
    s[2, 0, 0], s[2, 1, 1] = 1, -1
    g = torch.zeros((4, 4, 4), dtype=torch.complex128)
    for k in range(3):
        g[k, :2, 2:], g[k, 2:, :2] = -1j * s[k], 1j * s[k]
    g[3, :2, 2:] = g[3, 2:, :2] = torch.eye(2)
    return g.to(DEV)


class _Lattice:
    """D = 1 - kappa sum_mu w_mu [(1 - gamma_mu) U_mu(x) T_mu + (1 + gamma_mu) T_mu^dag U_mu^dag]."""

    def __init__(self, case, links):
        L = _dims(case)
        self.V, self.U, self.kappa = _vol(case), links, case["kappa"]
        self.w, bc = _wbc(case)
        s = torch.arange(self.V, device=DEV)
        self.c = [s % L[0], s // L[0] % L[1], s // (L[0] * L[1]) % L[2], s // (L[0] * L[1] * L[2])]
        st = (1, L[0], L[0] * L[1], L[0] * L[1] * L[2])
        self.up, self.dn, self.pu, self.pd = [], [], [], []
        for m in range(4):
            last, first = self.c[m] == L[m] - 1, self.c[m] == 0
            self.up.append(torch.where(last, s - (L[m] - 1) * st[m], s + st[m]))
            self.dn.append(torch.where(first, s + (L[m] - 1) * st[m], s - st[m]))
            self.pu.append(torch.where(last, float(bc[m]), 1.0).to(torch.float64)[:, None, None])
            self.pd.append(torch.where(first, float(bc[m]), 1.0).to(torch.float64)[:, None, None])
        self.g = _gammas()
        self.eye = torch.eye(4, device=DEV, dtype=torch.complex128)
        self.parity = (self.c[0] + self.c[1] + self.c[2] + self.c[3]) % 2

    def hop(self, psi, m, sign, dagger=False):
        """w_m (1 -/+ gamma_m) U T psi for sign +1, w_m (1 +/- gamma_m) T^dag U^dag psi for -1."""
        s = -1.0 if (sign > 0) != dagger else 1.0
        proj = (self.eye + s * self.g[m]) * self.w[m]
        if sign > 0:
            v = torch.matmul(psi[self.up[m]] * self.pu[m], self.U[m].transpose(1, 2))
        else:
            v = torch.matmul(psi, self.U[m].conj())[self.dn[m]] * self.pd[m]
        return torch.matmul(proj, v)

    def H(self, psi, dagger=False):
        out = torch.zeros_like(psi)
        for m in range(4):
            out += self.hop(psi, m, 1, dagger)
            out += self.hop(psi, m, -1, dagger)
        return out

    def D(self, psi, dagger=False):
        return psi - self.kappa * self.H(psi, dagger)

    def half_hop(self, psi, parity, dagger):
        """-kappa H_{parity, 1 - parity} on half-lattice fields."""
        full = torch.zeros((self.V, 4, 3), device=DEV, dtype=torch.complex128)
        full[self.parity == 1 - parity] = psi
        return -self.kappa * self.H(full, dagger)[self.parity == parity]

    def solve(self, b, dagger=False):
        """BiCGStab, restarted on the true residual until it no longer falls."""
        x = torch.zeros_like(b)
        dot = lambda a, c: torch.vdot(a.reshape(-1), c.reshape(-1))  # noqa: E731
        bn = torch.linalg.vector_norm(b)
        best = math.inf
        for _ in range(8):
            r = b - self.D(x, dagger)
            rn = float(torch.linalg.vector_norm(r) / bn)
            if rn < 2e-15 or rn > 0.5 * best:
                break
            best = rn
            r0, p, rho, e = r.clone(), r.clone(), dot(r, r), torch.zeros_like(b)
            goal = max(1e-15, 1e-11 * rn)
            for it in range(1500):
                v = self.D(p, dagger)
                a = rho / dot(r0, v)
                s = r - a * v
                t = self.D(s, dagger)
                om = dot(t, s) / dot(t, t)
                e = e + a * p + om * s
                r = s - om * t
                if it % 8 == 0 and float(torch.linalg.vector_norm(r) / bn) < goal:
                    break
                new = dot(r0, r)
                p = r + (new / rho) * (a / om) * (p - om * v)
                rho = new
            x = x + e
        return x


def _philox_gauss(seed, ids, V):
    """Complex-Gaussian fields of Philox4x32-10 (Salmon et al., SC'11): counter (site, component,
    vector, 0), key (seed low, seed high); two 53-bit uniforms, Box-Muller."""
    M = 0xFFFFFFFF
    out = []
    for v in ids:
        c0 = torch.arange(V, device=DEV, dtype=torch.int64)[:, None].expand(V, 12).contiguous()
        c1 = torch.arange(12, device=DEV, dtype=torch.int64)[None].expand(V, 12).contiguous()
        c2, c3 = torch.full_like(c0, int(v)), torch.zeros_like(c0)
        k0, k1 = seed & M, (seed >> 32) & M

        def mul(a, m):
            """(high, low) 32-bit words of a * m through 16-bit halves of m."""
            lo, hi = a * (m & 0xFFFF), a * (m >> 16)
            t = hi + (lo >> 16)
            return t >> 16, ((t & 0xFFFF) << 16) | (lo & 0xFFFF)

        for rnd in range(10):
            if rnd:
                k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
            h0, l0 = mul(c0, 0xD2511F53)
            h1, l1 = mul(c2, 0xCD9E8D57)
            c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        ua = ((c0 >> 5).double() * 67108864.0 + (c1 >> 6).double()) * 2.0 ** -53
        ub = ((c2 >> 5).double() * 67108864.0 + (c3 >> 6).double()) * 2.0 ** -53
        rho = torch.sqrt(-2.0 * torch.log1p(-ua))
        out.append(torch.polar(rho, 2.0 * math.pi * ub).reshape(V, 4, 3))
    return out


def _gmres(A, b, steps):
    """The minimiser of |b - A x| over the Krylov space of `steps` vectors."""
    V = [b / torch.linalg.vector_norm(b)]
    W = []
    for j in range(steps):
        w = A(V[j])
        W.append(w.reshape(-1))
        if j + 1 < steps:
            for _ in range(2):
                for v in V:
                    w = w - torch.vdot(v.reshape(-1), w.reshape(-1)) * v
            V.append(w / torch.linalg.vector_norm(w))
    Q, R = torch.linalg.qr(torch.stack(W, dim=1))
    y = torch.linalg.solve_triangular(R, (Q.mH @ b.reshape(-1))[:, None], upper=True)[:, 0]
    return sum(y[j] * V[j] for j in range(steps))


def _tiles(case):
    """Coarse site and local site of every fine site."""
    L, b = _dims(case), _block(case)
    s = torch.arange(_vol(case), device=DEV)
    c = [s % L[0], s // L[0] % L[1], s // (L[0] * L[1]) % L[2], s // (L[0] * L[1] * L[2])]
    C = [L[m] // b[m] for m in range(4)]
    q = [c[m] // b[m] for m in range(4)]
    e = [c[m] % b[m] for m in range(4)]
    return (q[0] + C[0] * (q[1] + C[1] * (q[2] + C[2] * q[3])),
            e[0] + b[0] * (e[1] + b[1] * (e[2] + b[2] * e[3])),
            C[0] * C[1] * C[2] * C[3], b[0] * b[1] * b[2] * b[3])


def _svd_left(A, k):
    """Leading k left singular vectors and values of a batch of tall matrices (rows x c)."""
    R = torch.eye(A.shape[-1], device=DEV, dtype=A.dtype).expand(A.shape[0], -1, -1)
    Q = A
    for _ in range(3):     # Cholesky QR, three times: Q orthonormal to rounding
        T = torch.linalg.cholesky(Q.mH @ Q).mH
        Q = torch.linalg.solve_triangular(T, Q, upper=True, left=False)
        R = T @ R
    u, s, _ = torch.linalg.svd(R)
    return Q @ u[:, :, :k], s[:, :k]


def _exact_svd(case, vec):
    coarse, local, d, nd = _tiles(case)
    k, r, n_s = case["k"], case["r"], case["n_s"]
    phi = None
    for s in range(n_s):
        T = torch.empty((d, 2, nd, 6, r), device=DEV, dtype=torch.complex128)
        for i in range(r):
            v = vec[s * r + i].to(torch.complex128).reshape(-1, 2, 6)
            T[coarse, 0, local, :, i] = v[:, 0]
            T[coarse, 1, local, :, i] = v[:, 1]
        T = T.reshape(2 * d, 6 * nd, r)
        A = T if phi is None else torch.cat([phi, T], dim=2)
        U, S = _svd_left(A, min(k, A.shape[2]))
        phi = U * S[:, None, :]
    q = U.sum(dim=1, keepdim=True)
    U = U * (q.conj() / q.abs())
    return U.mT.reshape(d, 2, k, 6 * nd).contiguous(), S.reshape(d, 2, k)


def _exact_galerkin(case, lat, P):
    coarse, local, d, nd = _tiles(case)
    b, k = _block(case), case["k"]
    Pt = P.reshape(2 * d, k, 6 * nd)
    X = torch.zeros((d, 2 * k, 2 * k), device=DEV, dtype=torch.complex128)
    Y = torch.zeros((8, d, 2 * k, 2 * k), device=DEV, dtype=torch.complex128)

    def project(f):        # P^dag f per aggregate: (d, 2k)
        T = torch.empty((d, 2, nd, 6), device=DEV, dtype=torch.complex128)
        f = f.reshape(-1, 2, 6)
        T[coarse, 0, local], T[coarse, 1, local] = f[:, 0], f[:, 1]
        return torch.einsum("tir,tr->ti", Pt.conj(), T.reshape(2 * d, -1)).reshape(d, 2 * k)

    for col in range(2 * k):
        a, i = col // k, col % k
        f = torch.zeros((_vol(case), 2, 6), device=DEV, dtype=torch.complex128)
        f[:, a] = P[:, a, i].reshape(d, nd, 6)[coarse, local]
        f = f.reshape(-1, 4, 3)
        X[:, :, col] += project(f)
        for m in range(4):
            for s, sign in enumerate((1, -1)):
                h = -lat.kappa * lat.hop(f, m, sign)
                cross = (lat.c[m] % b[m] == (b[m] - 1 if sign > 0 else 0))[:, None, None]
                X[:, :, col] += project(torch.where(cross, 0, h))
                Y[2 * m + s, :, :, col] += project(torch.where(cross, h, 0))
    return X, Y


def _exact_link_gradient(lat, g_b, x):
    lam = torch.zeros((8, 3, 3), device=DEV, dtype=torch.complex128)
    lam[0, 0, 1] = lam[0, 1, 0] = 1
    lam[1, 0, 1], lam[1, 1, 0] = -1j, 1j
    lam[2, 0, 0], lam[2, 1, 1] = 1, -1
    lam[3, 0, 2] = lam[3, 2, 0] = 1
    lam[4, 0, 2], lam[4, 2, 0] = -1j, 1j
    lam[5, 1, 2] = lam[5, 2, 1] = 1
    lam[6, 1, 2], lam[6, 2, 1] = -1j, 1j
    lam[7] = torch.diag(torch.tensor([1.0, 1.0, -2.0], device=DEV, dtype=torch.complex128)) / 3 ** 0.5
    out = torch.empty((4, lat.V, 8), device=DEV, dtype=torch.float64)
    for m in range(4):
        gu, xu = g_b[lat.up[m]], x[lat.up[m]]
        t1 = torch.matmul(lat.eye - lat.g[m], xu)
        t2 = torch.matmul(lat.eye + lat.g[m], x)
        for a in range(8):
            dU = torch.matmul(0.5j * lam[a], lat.U[m])
            v = ((g_b.conj() * torch.matmul(t1, dU.transpose(1, 2))).sum((1, 2)) +
                 (gu.conj() * torch.matmul(t2, dU.conj())).sum((1, 2)))
            out[m, :, a] = lat.kappa * lat.w[m] * (lat.pu[m][:, 0, 0] * v).real
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("dslash", "schur"):
        psi, links = _stencil_inputs(case, seed)
        lat = _Lattice(case, _widen(links))
        out = []
        for n in range(case["nrhs"]):
            v = _widen(psi[n])
            if kind == "schur":
                t = lat.half_hop(lat.half_hop(v, 1, case["dagger"]), 0, case["dagger"])
                v = v - t
            elif case["parity"] >= 0:
                v = lat.half_hop(v, case["parity"], case["dagger"])
            else:
                v = lat.D(v, case["dagger"])
            out.append(v if case["dtype"] in ("c128", "c64") else torch.view_as_real(v))
        return torch.stack(out)
    links, x = _mg_inputs(case, seed)
    if kind == "svd":
        return _exact_svd(case, x)
    lat = _Lattice(case, links)
    if kind == "vectors":
        r, s = case["r"], case["stream"]
        phis = _philox_gauss(_tv_seed(seed), range(s * r, s * r + r), _vol(case))
        return torch.stack([phi - _gmres(lat.D, lat.D(phi), 5) for phi in phis])
    if kind == "galerkin":
        return _exact_galerkin(case, lat, x)
    if kind == "solve":
        return torch.stack([lat.solve(b) for b in x])
    if kind == "step":
        return torch.stack([lat.solve(b) for b in x]), None
    sol = lat.solve(x[0])
    g_b = lat.solve(2.0 * sol, dagger=True)
    return sol[None], g_b[None], _exact_link_gradient(lat, g_b, sol)
